"""Transform kernels of the staged path at their edges: every channel-chunk width, tile groups that
are not full, zero points, float output, scales per channel, learnt matrices; on the path that
chooses by size (1) and on the one that always takes the tensor cores where it can (6)."""
import pytest

import wino_inputs as wi
from helpers import build_layer, per_channel
from test_gpu_parity import _compare

pytestmark = pytest.mark.gpu

SHAPES = [
    # N, C, H, W, K          chunks in / out
    (3, 96, 7, 9, 160),    # 96 / 80
    (2, 48, 6, 11, 96),    # 48 / 96
    (2, 80, 5, 5, 48),     # 80 / 48
    (1, 240, 6, 6, 144),   # 80 / 48, several chunks
    (1, 32, 1, 3, 16),     # 32 / 16, a group of one tile
]


@pytest.mark.parametrize("m", [2, 4, 6])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("variant", ["plain", "zero_points", "float_out", "per_channel_float", "flex"])
def test_chunks_and_options(m, shape, variant):
    N, C, H, W, K = shape
    L, x_q, w_q, bias = build_layer(wi.Workload("ch", 5400 + m, N, C, H, W, K, m, flex=variant == "flex"),
                                    out_dtype=1 if "float" in variant else 0)
    if variant == "zero_points":
        L.q_x.zero_point, L.q_w.zero_point, L.q_Y.zero_point = -9, 2, -5
    if variant.startswith("per_channel"):
        L = per_channel(L, 41 + m, spread=3.0)
    _compare(L, x_q, w_q, bias, 1)
    if variant in ("plain", "zero_points", "float_out"):
        _compare(L, x_q, w_q, bias, 6)


@pytest.mark.parametrize("m,N", [(2, 40), (4, 150), (6, 300)])
def test_several_units_per_block_on_the_tensor_cores(m, N):
    # more units than blocks, so that slots, accumulators and phases come round again
    L, x_q, w_q, bias = build_layer(wi.Workload("ch", 5500 + m, N, 128, 14, 15, 64, m))
    _compare(L, x_q, w_q, bias, 6)


@pytest.mark.parametrize("N", [592, 593, 887, 889])
def test_learnt_f6_around_one_wave_of_blocks(N):
    # one tile per image: the input and the output transform change kernels at 592 and 888 tiles
    L, x_q, w_q, bias = build_layer(wi.Workload("ch", 5600, N, 128, 6, 5, 128, 6, flex=True))
    _compare(L, x_q, w_q, bias, 1)
