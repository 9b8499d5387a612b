"""Which kernel wino_conv_forward takes, one launch or three, where the faster of the two is so by a margin
(microseconds of either beside each case, measured on B200)."""
import pytest

import wino_inputs as wi
from gpu_helpers import gpu_run
from helpers import build_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,H,W,K,m,options,launches", [
    (16, 512, 4, 4, 512, 4, {}, 3),                      # 9.9 / 8.8
    (16, 256, 8, 8, 256, 4, {}, 3),                      # 9.8 / 7.9
    (16, 128, 16, 16, 128, 6, {}, 3),                    # 11.4 / 9.1
    (2, 256, 8, 8, 256, 4, {}, 1),                       # 6.4 / 7.8
    (8, 128, 8, 8, 128, 2, {}, 1),                       # 4.8 / 7.2
    (16, 128, 14, 14, 128, 2, dict(q_M=False), 1),       # 10.1 / 14.2
    (16, 256, 8, 8, 256, 4, dict(q_M=False), 1),         # 9.8 / 11.5
    (32, 128, 8, 8, 128, 6, dict(q_M=False), 1),         # 10.7 / 15.0
    (16, 128, 14, 14, 128, 2, dict(flex=True), 3),       # 11.5 / 8.0
    (34, 128, 17, 17, 128, 2, dict(q_M=False), 3),       # 27.1 / 21.7
    (1, 512, 7, 4, 512, 4, dict(flex=True), 1),          # 7.1 / 9.8
    (16, 48, 16, 16, 80, 6, {}, 1),                      # 9.2 / 12.1
])
def test_one_launch_or_three(N, C, H, W, K, m, options, launches):
    options = dict(options)
    L, x_q, w_q, bias = build_layer(wi.Workload("d", 5800, N, C, H, W, K, m, flex=options.pop("flex", False)), **options)
    before = gpu_run(L, x_q, w_q, bias)
    assert before["launches"] == launches + 1            # and the weight transform
