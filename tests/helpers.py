"""Shared test helpers: build a layer statement (sizes, matrices, scales) for a
seeded workload.  Matrices and calibrated scales come from the oracle and are
handed to both sides as data."""
from __future__ import annotations

import copy

import numpy as np

import oracle
import wino_inputs as wi
from oracle import Layer, Quant
from oracle.calibrate import calibrate


def matrices(m: int, flex_seed: int | None = None):
    ct = oracle.cook_toom(m, wi.POINTS[m])
    BT, G, AT = ct["BT32"], ct["G32"], ct["AT32"]
    if flex_seed is not None:
        BT = wi.flex_perturb(BT, flex_seed, wi.S_BT)
        G = wi.flex_perturb(G, flex_seed, wi.S_G)
        AT = wi.flex_perturb(AT, flex_seed, wi.S_AT)
    return BT, G, AT


def build_layer(wl: wi.Workload, N: int | None = None, q_M: bool = True, out_dtype: int = 0,
                with_bias: bool = True, relu: bool = False):
    """Returns (Layer, x_q, w_q, bias) with every scale fixed."""
    x_q, s_x, w_q, s_w, bias = wi.make_tensors(wl, N=N, with_bias=with_bias)
    BT, G, AT = matrices(wl.m, wl.seed if wl.flex else None)
    L = Layer(N=x_q.shape[0], C=wl.C, H=wl.H, W=wl.W, K=wl.K, m=wl.m, BT=BT, G=G, AT=AT,
              out_dtype=out_dtype)
    L.q_x = Quant(scale=float(s_x))
    L.q_w = Quant(scale=float(s_w))
    L.q_M = Quant(enabled=1 if q_M else 0)
    if relu:
        L.q_Y = Quant(qmin=0)
    if wl.fixed_scales is not None:
        for q in (L.q_V, L.q_U, L.q_M, L.q_Y):
            q.scale = float(np.float32(wl.fixed_scales))
    else:
        L = calibrate(L, x_q, w_q, bias)
    return L, x_q, w_q, bias


def per_channel(L: Layer, seed: int, spread: float = 2.0) -> Layer:
    """Copy of L whose weight, transformed-weight, Hadamard-sum and output scales vary per output channel
    (the per-layer scale times a seeded factor in [1/spread, spread])."""
    f_w, f_U, f_M, f_Y = wi.channel_factors(seed, L.K, spread)
    P = copy.deepcopy(L)
    P.s_w_K = (np.float32(L.q_w.scale) * f_w).astype(np.float32)
    P.s_U_K = (np.float32(L.q_U.scale) * f_U).astype(np.float32)
    P.s_M_K = (np.float32(L.q_M.scale) * f_M).astype(np.float32) if L.q_M.enabled else None
    P.s_Y_K = (np.float32(L.q_Y.scale) * f_Y).astype(np.float32)
    return P


def small(wl: wi.Workload, **kw) -> wi.Workload:
    d = copy.copy(wl.__dict__)
    d.update(kw)
    return wi.Workload(**d)


def f6_order_sensitive(N: int, K: int, C: int = 64, H: int = 6, W: int = 6, out_dtype: int = 1):
    """An F6 layer whose output shows in which order A^T m A was summed: the codes of U, V and M are nearly
    all at or near their bounds, so that the sums of the six pixels that are not exact in fp32 exceed 24 bits.
    out_dtype 0 (whole 6x6 images, all alike): the output scale is 1/128 of the accumulators', a unit in the
    last place of a sum of 2^16 to 2^17, and channel k's bias takes its sum at pixel F6_ORDERED[k % 6] away."""
    L, x_q, w_q, bias = build_layer(wi.Workload("f6o", 5750 + K, N, C, H, W, K, 6), out_dtype=1)
    L.q_U.scale /= 3000.0
    L.q_V.scale /= 20.0
    # powers of two: nothing is lost in taking a bias to output codes
    L.q_M.scale = float(np.exp2(np.rint(np.log2(L.q_U.scale * L.q_V.scale * 127.0 * 127.0 * C ** 0.5 * 3e-3))))
    L.q_M.qmin = -128
    L.out_dtype = out_dtype
    if out_dtype == 0:
        assert (H, W) == (6, 6)
        x_q[:] = x_q[:1]
        L.q_Y.scale, L.q_Y.qmin = L.q_M.scale / 128.0, -128
        one = copy.deepcopy(L)
        one.N, one.out_dtype = 1, 1
        y = oracle.forward(one, x_q[:1], w_q, bias=None)[0]
        bias = np.array([-y[(*F6_ORDERED[k % 6], k)] for k in range(K)], np.float32)
    return L, x_q, w_q, bias


# (row, column) of the output pixels of an F6 tile whose sums need more than 24 bits
F6_ORDERED = [(4, 4), (3, 5), (5, 3), (4, 5), (5, 4), (5, 5)]
