"""The one-launch kernel for layers of few tiles (path 8) against the CPU oracle: edges of its
8-tile blocks, of its 16-channel output blocks and of the channel slices that the blocks of a
cluster split, every option, and the automatic choice at sizes around the point where it hands
over to the staged kernels."""
import numpy as np
import pytest

import oracle
import wino_inputs as wi
from helpers import build_layer, per_channel

pytestmark = pytest.mark.gpu

SMALL = 8


def _check(L, x_q, w_q, bias, path=SMALL):
    from gpu_helpers import gpu_run
    y_ref = oracle.forward(L, x_q, w_q, bias=bias)
    g = gpu_run(L, x_q, w_q, bias, path=path)
    if L.out_dtype == 0:
        bad = np.count_nonzero(g["y"] != y_ref)
    else:
        bad = np.count_nonzero(g["y"].view(np.uint32) != y_ref.view(np.uint32))
    assert bad == 0, f"y differs in {bad} of {y_ref.size}"
    return g


SHAPES = [
    # N, C, H, W, K
    (1, 4, 1, 1, 4),          # one tile, four output channels, a quarter of a copy
    (1, 16, 8, 8, 16),
    (1, 20, 7, 9, 24),        # channels in 4-byte pieces, half a block of outputs
    (2, 64, 13, 5, 20),       # four output channels more than a block
    (3, 68, 6, 6, 40),        # a slice of four channels behind a full one
    (1, 192, 9, 17, 36),
    (1, 512, 4, 4, 96),       # the most channels of F6: eight blocks a cluster
    (5, 128, 8, 8, 128),
]


@pytest.mark.parametrize("m", [2, 4, 6])
@pytest.mark.parametrize("shape", SHAPES)
def test_small_layer(m, shape):
    N, C, H, W, K = shape
    L, x_q, w_q, bias = build_layer(wi.Workload("sm", 5000 + m, N, C, H, W, K, m))
    g = _check(L, x_q, w_q, bias)
    assert g["path"] == SMALL and g["launches"] == 2     # the weight transform and the layer


@pytest.mark.parametrize("m", [2, 4, 6])
@pytest.mark.parametrize("variant", ["no_qm", "float_out", "no_qm_float", "relu", "no_bias", "zero_points", "flex",
                                     "per_channel", "saturating"])
def test_small_layer_variants(m, variant):
    L, x_q, w_q, bias = build_layer(wi.Workload("sv", 5100 + m, 2, 96, 7, 10, 48, m, flex=variant == "flex"),
                                    q_M=not variant.startswith("no_qm"), out_dtype=1 if "float" in variant else 0,
                                    relu=variant == "relu", with_bias=variant != "no_bias")
    if variant == "zero_points":
        L.q_x.zero_point, L.q_w.zero_point, L.q_Y.zero_point = 5, -3, 7
    if variant == "per_channel":
        L = per_channel(L, 31 + m, spread=3.0)
    if variant == "saturating":
        for q in (L.q_V, L.q_U, L.q_M, L.q_Y):
            q.scale = q.scale / 7.0
    _check(L, x_q, w_q, bias)


def test_products_beyond_16_bits_are_refused_and_still_computed():
    from paper_2002_10711_b200 import binding
    L, x_q, w_q, bias = build_layer(wi.Workload("sb", 5200, 1, 32, 6, 6, 32, 4))
    L.q_V.scale = float(np.float32(L.q_x.scale / 100.0))   # |v| / s_V reaches 1.3 million
    with pytest.raises(binding.WinoError) as e:
        binding.Plan.from_layer(L, path=SMALL)
    assert e.value.code == binding.ERR_UNSUPPORTED
    _check(L, x_q, w_q, bias, path=0)
    _check(L, x_q, w_q, bias, path=1)


@pytest.mark.parametrize("m,N", [(2, 1), (2, 24), (4, 2), (4, 40), (6, 3), (6, 60)])
def test_automatic_choice_on_both_sides_of_the_line(m, N):
    L, x_q, w_q, bias = build_layer(wi.Workload("sa", 5300 + m, N, 64, 11, 12, 96, m))
    _check(L, x_q, w_q, bias, path=0)


@pytest.mark.parametrize("m", [2, 4, 6])
@pytest.mark.parametrize("C", [16, 48])
def test_narrow_layers_of_many_tiles(m, C):
    # beyond 48 blocks the operands of narrow layers come by small copies instead of tensor copies
    L, x_q, w_q, bias = build_layer(wi.Workload("sn", 5600 + m, 9, C, 9 * m, 7 * m, 32, m))
    _check(L, x_q, w_q, bias)
