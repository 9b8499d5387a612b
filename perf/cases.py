"""The work that users of this library have it do, as cases to be timed and compared.

A case is a dict of plain values with a "kind":
  layer    one Winograd-aware convolution layer, forward (WinogradConv.forward)
  direct   one direct int8 3x3 convolution, stride 1 or 2 (binding.direct_conv_forward)
  weights  the weight transform of one layer (Plan.transform_weights), which a user pays on
           every weight update
  network  the sixteen 3x3 convolutions of a CIFAR-shaped ResNet-18 body chained layer by
           layer, stride-1 layers as Winograd layers of a per-layer tile size, stride-2
           layers as direct convolutions

Activations are post-ReLU-like half-normal codes, weights Gaussian codes, and the stage
scales fill the code ranges as a calibrated layer's do (they come from the variances of the
stages, which needs no pass over data).
"""
import math
import random

import numpy as np
import torch

from paper_2002_10711_b200 import binding, cook_toom
from paper_2002_10711_b200.layer import WinogradConv

SIGMA_X = 32.0                 # half-normal activation codes
RMS_W = 127.0 / 4.5            # Gaussian weight codes, the largest of a tensor at 127
S_X = 1.0 / 32.0
S_W = 0.05 * 4.5 / 127.0


def _layer(name, N, C, H, W, K, m, **options):
    c = dict(kind="layer", N=N, C=C, H=H, W=W, K=K, m=m, flex=False, per_channel=False, relu=True, bias=True,
             quantize_M=True, float_out=False, z_x=0)
    c.update(options)
    return dict(c, name=name)


def listed():
    return [
        # the smallest layer of the test configurations: one image, one call, latency
        _layer("layer_1x16x8x8_f2", 1, 16, 8, 8, 16, 2, relu=False),
        # one image through a wide late layer: a large weight tensor for a single tile column
        _layer("layer_1x512x4x4_f4", 1, 512, 4, 4, 512, 4),
        # a network's first stage at a training batch, narrow channels
        _layer("layer_64x64x32x32_f2", 64, 64, 32, 32, 64, 2, relu=False),
        # the headline layer of the benchmark
        _layer("layer_256x256x8x8_f4", 256, 256, 8, 8, 256, 4, relu=False),
        # learnt transforms, the large tile
        _layer("layer_128x128x16x16_f6_flex", 128, 128, 16, 16, 128, 6, flex=True, relu=False),
        # scales per output channel, ragged image, channel counts that are no powers of two
        _layer("layer_32x96x27x29_f4_per_channel", 32, 96, 27, 29, 160, 4, per_channel=True),
        # asymmetric activations into a head that wants real values
        _layer("layer_8x128x14x14_f4_zero_point_float", 8, 128, 14, 14, 64, 4, z_x=-9, float_out=True, relu=False),
        # the lossless candidate for the headline layer
        dict(kind="direct", name="direct_256x256x8x8_s1", N=256, C=256, H=8, W=8, K=256, stride=1),
        # a network's first layer, three channels in
        dict(kind="direct", name="direct_64x3x32x32_s1", N=64, C=3, H=32, W=32, K=64, stride=1),
        # weights of the widest layer after an update
        dict(kind="weights", name="weights_512x512_f4", C=512, K=512, m=4),
        # a whole network: one image, and the largest batch
        dict(kind="network", name="network_1", N=1, assignment=1005),
        dict(kind="network", name="network_256", N=256, assignment=1005),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# the largest listed case is the batch-256 network; a drawn single layer stays below these
_MOST_PIXEL_CHANNELS = 256 * 32 * 32 * 128
_MOST_MACS = 256 * 8 * 8 * 256 * 256 * 9


def _draw_layer(rng):
    widths = [16, 24, 32, 48, 64, 64, 96, 128, 128, 160, 192, 256, 256, 384, 512, 512]
    while True:
        N, C, K = _log_int(rng, 1, 256), rng.choice(widths), rng.choice(widths)
        if rng.random() < 0.5:
            K = C                                       # most layers of a residual network
        H = _log_int(rng, 4, 56)
        W = H if rng.random() < 0.6 else _log_int(rng, 4, 56)
        if N * H * W * (C + K) <= _MOST_PIXEL_CHANNELS and N * H * W * C * K * 9 <= _MOST_MACS:
            break
    c = _layer("", N, C, H, W, K, rng.choice([2, 4, 4, 6]))
    del c["name"]
    c["relu"] = rng.random() < 0.6
    c["bias"] = rng.random() < 0.7
    option = rng.random()
    if option < 0.12:
        c["flex"] = True
    elif option < 0.24:
        c["per_channel"] = True
    elif option < 0.32:
        c["float_out"], c["relu"] = True, False
    elif option < 0.40:
        c["z_x"] = rng.choice([-16, -9, 3, 7])
    elif option < 0.44:
        c["quantize_M"] = False
    return c


def _draw_direct(rng):
    if rng.random() < 0.25:
        while True:
            N, K, H = _log_int(rng, 1, 256), rng.choice([16, 32, 64]), _log_int(rng, 24, 64)
            if N * H * H * K <= 256 * 32 * 32 * 64:
                return dict(kind="direct", N=N, C=3, H=H, W=H, K=K, stride=rng.choice([1, 1, 2]))
    widths = [64, 128, 192, 256, 512]
    while True:
        N, C, K, stride = _log_int(rng, 1, 256), rng.choice(widths), rng.choice(widths), rng.choice([1, 2])
        H = _log_int(rng, 4, 56)
        W = H if rng.random() < 0.6 else _log_int(rng, 4, 56)
        # odd sizes at stride 2 cost several times more than even ones
        most = _MOST_MACS // (8 if stride == 2 and (H % 2 or W % 2) else 1)
        if N * H * W * (C + K) <= _MOST_PIXEL_CHANNELS and N * H * W * C * K * 9 <= most * stride * stride:
            return dict(kind="direct", N=N, C=C, H=H, W=W, K=K, stride=stride)


def draw(rng):
    kind = rng.random()
    if kind < 0.62:
        return _draw_layer(rng)
    if kind < 0.80:
        return _draw_direct(rng)
    if kind < 0.88:
        widths = [16, 32, 64, 96, 128, 192, 256, 384, 512]
        return dict(kind="weights", C=rng.choice(widths), K=rng.choice(widths), m=rng.choice([2, 4, 6]))
    return dict(kind="network", N=_log_int(rng, 1, 256), assignment=rng.randrange(1 << 16))


# --- the ResNet-18 body ------------------------------------------------------------------
def _network_layers(case):
    """(C, size, K, stride, m) of the sixteen convolutions."""
    rng = random.Random(case["assignment"])
    out, cin, size = [], 64, 32
    for stage, width in enumerate([64, 128, 256, 512]):
        for i in range(4):
            stride = 2 if stage > 0 and i == 0 else 1
            out.append((cin, size, width, stride, rng.choice([2, 4, 6])))
            size //= stride
            cin = width
    return out


# --- inputs ------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _activations(gen, shape, z_x=0):
    v = torch.randn(shape, generator=gen, device="cuda").mul_(SIGMA_X).abs_().round_()
    return v.add_(z_x).clamp_(-127, 127).to(torch.int8)


def _weights(gen, K, C):
    return torch.randn((K, 3, 3, C), generator=gen, device="cuda").mul_(RMS_W).round_().clamp_(-127, 127).to(torch.int8)


def _stage_scales(BT, G, AT, C, s_x, mean_square_x, mean_x):
    """Scales (V, U, M, Y) that put four to five standard deviations of each stage on 127."""
    BT, G, AT = (np.asarray(a, np.float64) for a in (BT, G, AT))
    b2, b1, g2, a2 = (BT ** 2).sum(1), BT.sum(1), (G ** 2).sum(1), AT ** 2
    V2 = np.outer(b2, b2) * (mean_square_x - mean_x ** 2) + (np.outer(b1, b1) * mean_x) ** 2
    U2 = np.outer(g2, g2) * RMS_W ** 2
    s_V = s_x * 4.0 * math.sqrt(V2.max()) / 127.0
    s_U = S_W * 4.0 * math.sqrt(U2.max()) / 127.0
    M2 = C * V2 * s_x ** 2 * U2 * S_W ** 2
    s_M = 4.5 * math.sqrt(M2.max()) / 127.0
    s_Y = 4.5 * math.sqrt((a2 @ M2 @ a2.T).max()) / 127.0
    return tuple(float(np.float32(s)) for s in (s_V, s_U, s_M, s_Y))


def _make_layer(gen, rng, N, C, H, W, K, m, s_x, mean_square_x, mean_x, flex=False, per_channel=False, relu=True,
                bias=True, quantize_M=True, float_out=False, z_x=0):
    """The plan of one layer with its transformed weights; returns (WinogradConv, s_Y)."""
    BT, G, AT = cook_toom(m)
    if flex:
        BT, G, AT = ((a + 0.01 * rng.standard_normal(a.shape)).astype(np.float32) for a in (BT, G, AT))
    s_V, s_U, s_M, s_Y = _stage_scales(BT, G, AT, C, s_x, mean_square_x, mean_x)
    plan = binding.Plan(N, C, H, W, K, m, BT, G, AT, dict(scale=s_x, zero_point=z_x), dict(scale=S_W),
                        dict(scale=s_V), dict(scale=s_U), dict(scale=s_M, enabled=int(quantize_M)),
                        dict(scale=s_Y, qmin=0 if relu else -127), out_dtype=int(float_out))
    if per_channel:
        factors = np.exp(rng.uniform(-math.log(2.0), math.log(2.0), (3, K)))
        plan.set_channel_scales((S_W * factors[0]).astype(np.float32), (s_U * factors[1]).astype(np.float32),
                                (s_M * factors[2]).astype(np.float32), None)
    conv = WinogradConv(plan)
    b = (torch.randn(K, generator=gen, device="cuda") * (s_Y * 7.0)) if bias else None
    conv.load_weights(_weights(gen, K, C), b)
    return conv, s_Y


def _direct_scale(C, s_x, mean_square_x):
    return float(np.float32(4.5 * math.sqrt(9.0 * C * mean_square_x) * RMS_W * s_x * S_W / 127.0))


HALF_NORMAL = (SIGMA_X ** 2, SIGMA_X * math.sqrt(2.0 / math.pi))   # mean square, mean
AFTER_RELU = (0.5 * (127.0 / 4.5) ** 2, 127.0 / 4.5 / math.sqrt(2.0 * math.pi))


def prepare(case, seed):
    gen, rng = _generator(seed), np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "layer":
        options = {k: case[k] for k in ("flex", "per_channel", "relu", "bias", "quantize_M", "float_out", "z_x")}
        N, C, H, W, K, m = (case[k] for k in ("N", "C", "H", "W", "K", "m"))
        conv, _ = _make_layer(gen, rng, N, C, H, W, K, m, S_X, *HALF_NORMAL, **options)
        return dict(kind=kind, conv=conv, x=_activations(gen, (N, H, W, C), case["z_x"]))
    if kind == "direct":
        N, C, H, W, K, stride = (case[k] for k in ("N", "C", "H", "W", "K", "stride"))
        s_Y = _direct_scale(C, S_X, HALF_NORMAL[0])
        Ho, Wo = (H - 1) // stride + 1, (W - 1) // stride + 1
        return dict(kind=kind, sizes=(N, C, H, W, K, stride), q_x=dict(scale=S_X), q_w=dict(scale=S_W),
                    q_Y=dict(scale=s_Y, qmin=0), x=_activations(gen, (N, H, W, C)), w=_weights(gen, K, C),
                    bias=torch.randn(K, generator=gen, device="cuda") * (s_Y * 7.0),
                    y=torch.empty((N, Ho, Wo, K), dtype=torch.int8, device="cuda"))
    if kind == "weights":
        C, K, m = case["C"], case["K"], case["m"]
        BT, G, AT = cook_toom(m)
        s_V, s_U, s_M, s_Y = _stage_scales(BT, G, AT, C, S_X, *HALF_NORMAL)
        plan = binding.Plan(16, C, 8, 8, K, m, BT, G, AT, dict(scale=S_X), dict(scale=S_W), dict(scale=s_V),
                            dict(scale=s_U), dict(scale=s_M), dict(scale=s_Y))
        return dict(kind=kind, plan=plan, w=_weights(gen, K, C),
                    Uq=torch.empty(plan.weight_bytes, dtype=torch.int8, device="cuda"))
    N, steps, s_x, moments = case["N"], [], S_X, HALF_NORMAL
    x = _activations(gen, (N, 32, 32, 64))
    for C, size, K, stride, m in _network_layers(case):
        if stride == 1:
            conv, s_Y = _make_layer(gen, rng, N, C, size, size, K, m, s_x, *moments)
            steps.append(dict(conv=conv, y=conv.empty_output()))
        else:
            s_Y = _direct_scale(C, s_x, moments[0])
            steps.append(dict(conv=None, sizes=(N, C, size, size, K, stride), q_x=dict(scale=s_x),
                              q_w=dict(scale=S_W), q_Y=dict(scale=s_Y, qmin=0), w=_weights(gen, K, C),
                              y=torch.empty((N, size // 2, size // 2, K), dtype=torch.int8, device="cuda")))
        s_x, moments = s_Y, AFTER_RELU
    return dict(kind=kind, x=x, steps=steps)


# --- one pass ----------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "layer":
        return state["conv"].forward(state["x"])
    if kind == "direct":
        binding.direct_conv_forward(*state["sizes"], state["q_x"], state["q_w"], state["q_Y"], state["x"],
                                    state["w"], state["bias"], state["y"])
        return state["y"]
    if kind == "weights":
        state["plan"].transform_weights(state["w"], state["Uq"])
        return state["Uq"]
    x, outputs = state["x"], []
    for step in state["steps"]:
        if step["conv"] is not None:
            step["conv"].forward(x, step["y"])
        else:
            binding.direct_conv_forward(*step["sizes"], step["q_x"], step["q_w"], step["q_Y"], x, step["w"], None,
                                        step["y"])
        x = step["y"]
        outputs.append(x)
    return outputs


# --- what a pass cannot do without -------------------------------------------------------
def _layer_work(N, C, H, W, K, m, out_bytes=1):
    t2, tiles = (m + 2) ** 2, N * -(-H // m) * -(-W // m)
    return dict(bytes=N * H * W * (C + K * out_bytes) + t2 * K * C + 4 * K, flops=2 * t2 * tiles * C * K)


def _direct_work(N, C, H, W, K, stride):
    out = N * ((H - 1) // stride + 1) * ((W - 1) // stride + 1)
    return dict(bytes=N * H * W * C + out * K + 9 * K * C + 4 * K, flops=2 * out * 9 * C * K)


def work(case):
    kind = case["kind"]
    if kind == "layer":
        return _layer_work(*(case[k] for k in ("N", "C", "H", "W", "K", "m")), 4 if case["float_out"] else 1)
    if kind == "direct":
        return _direct_work(*(case[k] for k in ("N", "C", "H", "W", "K", "stride")))
    if kind == "weights":
        C, K, t = case["C"], case["K"], case["m"] + 2
        return dict(bytes=K * C * (9 + t * t), flops=2 * K * C * (9 * t + 3 * t * t))
    parts = [_layer_work(case["N"], C, size, size, K, m) if stride == 1
             else _direct_work(case["N"], C, size, size, K, stride)
             for C, size, K, stride, m in _network_layers(case)]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def tolerance(case):
    # integer codes are the same bytes whatever the implementation; real-valued outputs are
    # sums of at most 64 products in 32-bit floats
    if case["kind"] == "layer" and case["float_out"]:
        return {"rel": 1e-5}
    return "exact"
