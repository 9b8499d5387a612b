"""Direct convolution: at most four input channels (window in registers), and odd image sizes at
stride 2 on the tensor cores, against the oracle's integer convolution."""
import numpy as np
import pytest

import oracle
import wino_inputs as wi
from oracle import Quant
from test_gpu_direct import _run

pytestmark = pytest.mark.gpu


def _check(N, C, H, W, K, stride, zero_points=False, out_dtype=0):
    x_q = wi.uniform_int8(6000 + C, 1, (N, H, W, C), -128, 127)
    w_q, s_w = wi.gaussian_weight_codes(6000 + K, 2, (K, 3, 3, C), 0.05)
    s_x = float(np.float32(1 / 32))
    z_x, z_w = (7, -5) if zero_points else (0, 0)
    bias = wi.bias_values(6000, 3, K, 0.5)
    acc = oracle.direct_conv_i32(x_q, w_q, z_x=z_x, z_w=z_w, stride=stride)
    s_in = s_x * float(s_w)
    q_Y = Quant(scale=float(np.float32(float(np.abs(acc).max()) * s_in / 127.0)), zero_point=3 if zero_points else 0)
    got = _run(N, C, H, W, K, stride, Quant(scale=s_x, zero_point=z_x), Quant(scale=float(s_w), zero_point=z_w), q_Y,
               x_q, w_q, bias, out_dtype=out_dtype)
    if out_dtype == 0:
        assert (got == oracle.requantize_acc(acc, s_in, q_Y, bias)).all()
    else:
        want = acc.astype(np.float64) * np.float64(np.float32(s_in)) + bias.astype(np.float64)
        assert np.abs(got - want).max() <= 1e-6 * np.abs(want).max()
    from paper_2002_10711_b200 import binding
    assert binding.direct_last_status() == 0


@pytest.mark.parametrize("C", [1, 2, 3, 4])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 9, 13, 16), (1, 32, 8, 33), (3, 7, 30, 67)])   # N, H, W, K
@pytest.mark.parametrize("stride,zero_points,out_dtype", [(1, False, 0), (2, True, 0), (1, True, 1)])
def test_narrow_input(C, shape, stride, zero_points, out_dtype):
    N, H, W, K = shape
    _check(N, C, H, W, K, stride, zero_points, out_dtype)


@pytest.mark.parametrize("shape", [(1, 64, 1, 1, 32), (3, 128, 9, 9, 64), (5, 64, 33, 8, 96), (2, 192, 6, 17, 256),
                                   (9, 64, 5, 3, 64), (1, 64, 255, 1, 32)])
def test_odd_sizes_at_stride_two(shape):
    _check(*shape, 2)


def test_many_pixels_per_warp():
    _check(40, 3, 61, 33, 70, 1)     # more groups of 32 pixels than warps, two blocks of channels
