"""The layer with which the GPU tests tell ordered from factored sums in F6's output transform does tell them
apart: an fp32 model of the kernels' two passes agrees with the oracle bit for bit when the six pixels are summed
in the oracle's order, and differs from it in every one of the six when they are factored like the others."""
import numpy as np
import pytest

import oracle
from helpers import F6_ORDERED, f6_order_sensitive

f32 = np.float32


def _fma(c, a, b):
    # exact in double (multiples of 2^-10 below 2^20), rounded once
    return (np.float64(c) * a.astype(np.float64) + b.astype(np.float64)).astype(f32)


def _pass(m, ordered):
    s1, d1, s2, d2, s3, d3 = m[1] + m[2], m[1] - m[2], m[3] + m[4], m[3] - m[4], m[5] + m[6], m[5] - m[6]

    def row(p, first, second):   # rows 3, 4 and 5: 2^p and 2^-p
        if row_is_ordered[p]:
            sign = 1.0 if p == 4 else -1.0
            return _fma(sign * 2.0 ** -p, m[6], _fma(2.0 ** -p, m[5], _fma(sign * 2.0 ** p, m[4], _fma(2.0 ** p, m[3], first))))
        return _fma(2.0 ** -p, second[1], _fma(2.0 ** p, second[0], first))

    row_is_ordered = {p: ordered(p) for p in (3, 4, 5)}
    return [m[0] + s1 + s2 + s3, _fma(0.5, d3, _fma(2.0, d2, d1)), _fma(0.25, s3, _fma(4.0, s2, s1)),
            row(3, d1, (d2, d3)), row(4, s1, (s2, s3)), row(5, d1, (d2, d3)) + m[7]]


def _model(m_q, ordered_pixels):
    """A^T m A of every tile and channel, [6][6][T][K]."""
    m = m_q.astype(f32).reshape(8, 8, *m_q.shape[1:])
    R = [_pass(list(m[i]), lambda a: False) for i in range(8)]
    cols = [_pass([R[i][b] for i in range(8)], lambda a, b=b: (a, b) in ordered_pixels) for b in range(6)]
    return np.array([[cols[b][a] for b in range(6)] for a in range(6)])


def test_the_two_orders_differ_in_every_ordered_pixel():
    L, x_q, w_q, _ = f6_order_sensitive(40, 128)
    y, d = oracle.forward(L, x_q, w_q, bias=None, dumps=True)
    image = lambda Y: (np.moveaxis(Y, 2, 0) * f32(L.q_M.scale)).astype(f32)   # one tile per image
    assert (image(_model(d["m_q"], F6_ORDERED)).view(np.uint32) == y.view(np.uint32)).all()
    for p in F6_ORDERED:
        other = image(_model(d["m_q"], [q for q in F6_ORDERED if q != p]))
        assert (other[:, p[0], p[1]] != y[:, p[0], p[1]]).any(), p
    assert (image(_model(d["m_q"], [])) != y).any(axis=(0, 3)).sum() == len(F6_ORDERED)


@pytest.mark.parametrize("K", [64, 128])
def test_the_two_orders_differ_in_codes(K):
    L, x_q, w_q, bias = f6_order_sensitive(1, K, out_dtype=0)
    y, d = oracle.forward(L, x_q, w_q, bias=bias, dumps=True)

    def codes(Y):
        real = _fma(f32(128.0), np.moveaxis(Y, 2, 0), (bias / f32(L.q_Y.scale))[None, None, None])
        return np.clip(np.rint(real), -128, 127).astype(np.int8)

    assert (codes(_model(d["m_q"], F6_ORDERED)) == y).all()
    assert (codes(_model(d["m_q"], [])) != y).any()
