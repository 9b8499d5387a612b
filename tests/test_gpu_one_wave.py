"""The GEMM's two quantizers of int8 codes (chosen by the width of a block's columns), and transform
builds that are chosen by whether all blocks of a grid are resident at once, on both sides of each line."""
import numpy as np
import pytest
import torch

import oracle
import wino_inputs as wi
from helpers import build_layer, f6_order_sensitive, per_channel
from paper_2002_10711_b200 import binding
from paper_2002_10711_b200.layer import WinogradConv
from test_gpu_parity import _compare

pytestmark = pytest.mark.gpu


# blocks of 256 output channels (saturating pack) and narrower ones (clamp on 16-bit lanes), these with one, two
# and four 128-tile blocks to an accumulator; bounds other than 127
@pytest.mark.parametrize("N,C,K", [(6, 128, 256), (6, 64, 96), (120, 64, 192), (360, 64, 64), (720, 32, 64),
                                   (360, 64, 128)])
@pytest.mark.parametrize("variant", ["plain", "relu", "per_channel", "zero_point_y", "saturating", "bound_100"])
def test_quantizers_of_the_gemm(N, C, K, variant):
    L, x_q, w_q, bias = build_layer(wi.Workload("oc", 5720, N, C, 9, 11, K, 4), relu=variant == "relu")
    if variant == "per_channel":
        L = per_channel(L, 43, spread=3.0)
    if variant == "zero_point_y":
        L.q_Y.zero_point = -11
    if variant == "saturating":
        for q in (L.q_V, L.q_U, L.q_M, L.q_Y):
            q.scale = q.scale / 7.0
    if variant == "bound_100":
        L.q_M.qmin, L.q_M.qmax = -100, 100
    _compare(L, x_q, w_q, bias, 1)


# rounded products up to the limit of the 16-bit lanes: inputs and weights of +-127, V and U codes nearly all
# at their bounds, scales just inside the bounds that the plan checks (|B^T| row sums 2, 10; |V| <= 128 row^2)
@pytest.mark.parametrize("m,row", [(2, 2), (4, 10)])
def test_products_at_the_limit_of_16_bits(m, row):
    L, x_q, w_q, bias = build_layer(wi.Workload("lim", 5760 + m, 9, 16, 13, 15, 64, m))
    x_q = np.where(x_q > np.median(x_q), 127, -127).astype(np.int8)
    w_q = np.where(w_q > 0, 127, -127).astype(np.int8)
    L.q_V.scale = L.q_x.scale * (128.0 * row * row) / 31990.0
    L.q_U.scale = L.q_w.scale / 100.0
    L.q_M.scale = L.q_U.scale * L.q_V.scale * (16384.0 * 16) / 31990.0
    for path in (1, 6):
        _compare(L, x_q, w_q, bias, path)


# blocks per SM x 148: 12, 14 and 16 in F4 (input; 16 also output), 7 in F6
@pytest.mark.parametrize("m,N", [(4, 1776), (4, 1777), (4, 2072), (4, 2073), (4, 2368), (4, 2369), (6, 1036), (6, 1037)])
def test_around_one_wave_of_blocks(m, N):
    # one tile per image and 128 channels: blocks = images
    L, x_q, w_q, bias = build_layer(wi.Workload("ow", 5700 + m, N, 128, m, m - 1, 128, m))
    _compare(L, x_q, w_q, bias, 1)


# one to nine blocks of a transform per SM: from two to eight the grid asks for the shared memory that
# spreads it over the SMs, the output's only where the GEMM's items are level
@pytest.mark.parametrize("m", [2, 4, 6])
@pytest.mark.parametrize("N", [148, 149, 296, 512, 1184, 1185])
def test_few_blocks_per_sm(m, N):
    L, x_q, w_q, bias = build_layer(wi.Workload("fb", 5770 + m, N, 128, m, m - 1, 128, m))
    _compare(L, x_q, w_q, bias, 1)


# F6 output, one tile per image: one channel per thread up to 592 blocks of 128 and 888 of 64 channels, pairs
# from there on; blocks at most one, and more, to an SM; codes at their bounds, where the factored sums are largest
@pytest.mark.parametrize("K,N", [(128, 148), (128, 149), (128, 592), (128, 593), (64, 592), (64, 593), (64, 888),
                                 (64, 889), (96, 50)])
@pytest.mark.parametrize("variant", ["plain", "saturating", "float_out"])
def test_f6_output_transform(K, N, variant):
    L, x_q, w_q, bias = build_layer(wi.Workload("o6", 5750 + K, N, 64, 6, 5, K, 6),
                                    out_dtype=1 if variant == "float_out" else 0)
    if variant == "saturating":
        L.q_M.scale, L.q_M.qmin = L.q_M.scale / 1000.0, -128
    _compare(L, x_q, w_q, bias, 1)
    _compare(L, x_q, w_q, bias, 8, dumps=False)


# the same builds, and the one-launch kernel, on sums that show the order of their terms: as floats, and as codes
# of a unit in the last place each (the one-channel builds write codes only)
@pytest.mark.parametrize("K,N", [(128, 148), (128, 149), (128, 592), (128, 593), (64, 592), (64, 593), (64, 888),
                                 (64, 889), (96, 50)])
@pytest.mark.parametrize("out", ["codes", "float", "float_ragged"])
def test_f6_output_transform_sums_in_order(K, N, out):
    if out == "float_ragged":
        L, x_q, w_q, bias = f6_order_sensitive((N + 3) // 4, K, H=11, W=12)
    else:
        L, x_q, w_q, bias = f6_order_sensitive(N, K, out_dtype=0 if out == "codes" else 1)
    _compare(L, x_q, w_q, bias, 1)
    _compare(L, x_q, w_q, bias, 8, dumps=False)


# F6 output: the line between its two builds is another with scales per output channel; a plan that has run
# takes them, and loses them again, with tensor maps of the build that it then runs
@pytest.mark.parametrize("K,N", [(128, 296), (128, 297), (64, 400)])
def test_f6_channel_scales_on_a_plan_that_has_run(K, N):
    L, x_q, w_q, bias = build_layer(wi.Workload("o6c", 5780 + K, N, 64, 6, 5, K, 6))
    P = per_channel(L, 47)
    conv = WinogradConv(binding.Plan.from_layer(L, path=1))
    x = torch.from_numpy(x_q).cuda()
    for layer, scales in ((L, None), (P, (P.s_w_K, P.s_U_K, P.s_M_K, P.s_Y_K)), (L, (None,) * 4)):
        if scales is not None:
            conv.plan.set_channel_scales(*scales)
        conv.load_weights(w_q, bias)
        y = conv.forward(x)
        assert conv.plan.last_status() == 0
        assert (y.cpu().numpy() == oracle.forward(layer, x_q, w_q, bias=bias)).all()


# several tiles a block (64, 32 and 16 channels a chunk), one channel per thread and two
@pytest.mark.parametrize("m,C", [(4, 64), (4, 32), (4, 16), (6, 64), (6, 32)])
@pytest.mark.parametrize("N", [1, 37, 700])
def test_narrow_chunks_around_one_wave(m, C, N):
    L, x_q, w_q, bias = build_layer(wi.Workload("on", 5710 + m, N, C, 2 * m, 2 * m - 1, 32, m))
    _compare(L, x_q, w_q, bias, 1)


@pytest.mark.parametrize("m", [2, 4, 6])
@pytest.mark.parametrize("variant", ["plain", "zero_points", "flex", "float_out"])
def test_chunks_of_112_channels(m, variant):
    L, x_q, w_q, bias = build_layer(wi.Workload("o7", 5730 + m, 3, 112, 7, 9, 224, m, flex=variant == "flex"),
                                    out_dtype=1 if variant == "float_out" else 0)
    if variant == "zero_points":
        L.q_x.zero_point, L.q_w.zero_point, L.q_Y.zero_point = -9, 2, -5
    _compare(L, x_q, w_q, bias, 1)


# stages of 64 channels, full and not, under accumulators of four, two and one 128-tile blocks; the
# last group of tiles ragged; at least five items to each of 148 blocks, so that the four stages come round again
@pytest.mark.parametrize("C", [16, 32, 48, 64])
@pytest.mark.parametrize("K,N,blocks", [(64, 1793, 4), (96, 801, 1), (128, 801, 2)])
def test_narrow_stages_of_the_gemm(C, K, N, blocks):
    L, x_q, w_q, bias = build_layer(wi.Workload("ns", 5740 + C, N, C, 11, 9, K, 6))
    assert 64 * -(-4 * N // (128 * blocks)) >= 5 * 148
    _compare(L, x_q, w_q, bias, 1)
