"""The FP64 evaluation of csrc/boys_region.cuh (start, eval_regular), modelled with
Python integers operation by operation, on the tables that csrc/gen_local.py
generates, against exact rational arithmetic on the printed coefficients: the
anchors r_{A,k}, what the upward recurrence makes of r_B, and the asymptotic form,
each followed by its own recurrence of the paper's Algorithm 1 (downward in A,
upward in B and C) in 400-bit fixed point.

Derived bounds, relative to F_k: a product drops at most 3 units of its last place
and the tables' low terms at most 3 x 2^5 units of a value of at least 2^61.9
(2^-55.3); a step adds two products on sums of at least 2^56.9 units
(2 x 3 x 2^-56.9, of which later steps keep a part below one, since all terms are
positive) and region C's anchors an interpolation error below 2^-60.  Sixteen of
the steps' errors at once would be 2^-50.3; the bound here is 2^-53, FP64's own
half-ulp rounding (the largest seen is 2^-53.9), and 3e-17 absolute in A and B.
"""
import importlib.util
import math
import os
import struct

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_10059_gb300", "csrc")
X0, X1 = 11.899848152108484, 28.989337738820740
M64 = (1 << 64) - 1
W = 400


def _gen():
    spec = importlib.util.spec_from_file_location("gen_local", os.path.join(CSRC, "gen_local.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


GEN = _gen()
TABLE, EXP = GEN.table(), GEN.exp_coeffs()
RB_P, RB_Q, RA_P, RA_Q = GEN._rationals()


def _mulhi(a, b, add=0):
    assert 0 <= a <= M64 and 0 <= b <= M64
    a0, a1, b0, b1 = a & 0xFFFFFFFF, a >> 32, b & 0xFFFFFFFF, b >> 32
    r = a1 * b1 + ((a1 * b0) >> 32) + ((a0 * b1) >> 32) + add
    assert r <= M64
    return r


def _model(K, x):
    """{order: (significand, exponent)}, value significand 2^exponent, before the cut to a double."""
    xb = struct.unpack("<Q", struct.pack("<d", x))[0]
    m, be = ((xb << 11) | 1 << 63) & M64, xb >> 52
    X, q = m >> max(1027 - be, 0) if be > 900 else 0, max(be - 1027, 0)
    vh, in_c = X >> 32, x >= X1
    if in_c:
        vh &= 0x7FFFFFFF | (be << 31) & 0xFFFFFFFF
    bits = (9 if K <= 12 else 10) if in_c else 9
    h = (be - 1023) >> 1 if in_c else 0
    e = TABLE[K][(465 if in_c else int(x >= X0)) + (vh >> (32 - bits))]
    t = ~((vh << 32 | X & 0xFFFFFFFF) << bits) & M64
    t32 = t >> 32
    b, n, eb, w = e[:8], e[8] - h * (2 * K + 1), e[9], e[10]
    u5 = b[5] + ((t32 * (b[6] + ((t32 * b[7]) >> 32))) >> 32)
    assert u5 < 1 << 32
    y = b[4] + (((t32 * u5) >> 32) << 5)
    for i in (3, 2, 1, 0):
        y = _mulhi(t, y, b[i])
    e5 = EXP[5] + ((t32 * (EXP[6] + ((t32 * EXP[7]) >> 32))) >> 32)
    E = EXP[4] + (((t32 * e5) >> 32) << 5)
    for i in (3, 2, 1, 0):
        E = _mulhi(t, E, EXP[i])
    Em = _mulhi(w, E)
    out = {}

    def normalise(y, n, gain):
        assert 1 << 32 <= y < 1 << 63
        lead = (y >> 32).bit_length() - 1
        return y << (30 - lead), n + lead + gain - 30

    y, n = normalise(y, n, 0)
    out[K] = (y, eb + n + 1 - 1023 - 62)
    for l in range(K - 1, -1, -1):
        assert n >= 0
        T = _mulhi(X, y, Em >> n)
        assert (1 << 56) < T < 0.56 * 2 ** 64
        s = (2 * l + 1).bit_length() - 1
        y, gain = (T, 6) if l == 0 else (_mulhi(T, (1 << (63 + s)) // (2 * l + 1)), 7 - s)
        y, n = normalise(y, n + q, gain)
        out[l] = (y, eb + n + 1 - 1023 - 62)
    return out


def _fix(v):
    n, d = float(v).as_integer_ratio()
    return (n << W) // d


def _poly(c, x):
    v = 0
    for a in reversed(c):
        v = ((v * x) >> W) + _fix(a)
    return v


def _exp_neg(x):
    s = term = 1 << W  # e^{-x} = (e^{-x/64})^64
    i = 0
    while term:
        i += 1
        term = (term * x >> W) // (64 * i)
        s += -term if i & 1 else term
    for _ in range(6):
        s = s * s >> W
    return s


def _algorithm1(K, x):
    xf = _fix(x)
    if x < X0:
        f, e = [0] * (K + 1), _exp_neg(xf)
        f[K] = (_poly(RA_P[K], xf) << W) // _poly(RA_Q[K], xf)
        for l in range(K - 1, -1, -1):
            f[l] = ((2 * xf * f[l + 1] >> W) + e) // (2 * l + 1)
        return f
    if x < X1:
        f, e = [(_poly(RB_P, xf) << W) // _poly(RB_Q, xf)], _exp_neg(xf)
    else:
        pi = 0
        for mul, d in ((16, 5), (-4, 239)):
            t, i, sign = (1 << W) // d, 1, 1
            while t:
                pi += sign * mul * (t // i)
                t, i, sign = t // (d * d), i + 2, -sign
        f, e = [(math.isqrt(pi << W) // 2 << W) // math.isqrt(xf << W)], 0
    for l in range(K):
        f.append((((2 * l + 1) * f[l] - e) << W) // (2 * xf))
    return f


def _points(K):
    """Interval edges and their neighbours in every region, the ends of the
    regions, tiny and large arguments."""
    pts = [0.0, 5e-324, 1e-300, 2.0 ** -60, 1e-9, X0, math.nextafter(X0, 0), math.nextafter(X0, 99), X1,
           math.nextafter(X1, 0), math.nextafter(X1, 99), 2.0 ** 28, 31.999, 32.0, 63.99, 64.0, 1e4, 3.3e7]
    for j in (1, 7, 64, 150, 190, 191, 255, 300, 463):
        pts += [j / 16, math.nextafter(j / 16, 0), math.nextafter(j / 16, 99), (j + 0.5 + K / 70) / 16]
    return pts + [30.0 * 1.61 ** i for i in range(12)]


@pytest.mark.parametrize("K", [0, 1, 2, 3, 5, 8, 12, 13, 20, 32])
def test_model_against_exact_algorithm1(K):
    for x in _points(K):
        got, ref = _model(K, x), _algorithm1(K, x)
        for l in range(K + 1):
            y, ex = got[l]
            v = y << (W + ex) if W + ex >= 0 else y >> -(W + ex)
            err = abs(v - ref[l])
            assert err << 53 <= ref[l], (K, l, x, math.log2(err / ref[l]))
            assert x >= X1 or err / (1 << W) <= 3e-17, (K, l, x)


def test_planted_mistakes_fail():
    """One unit in an anchor's exponent, a table entry of the neighbouring
    interval, and kappa of the next order are each far outside the bound."""
    got, ref = _model(5, 3.3), _algorithm1(5, 3.3)
    y, ex = got[2]
    assert abs((y << (W + ex + 1)) - ref[2]) << 53 > ref[2]
    keep = TABLE[5][52]
    TABLE[5][52] = TABLE[5][53]
    try:
        y, ex = _model(5, 3.3)[5]
    finally:
        TABLE[5][52] = keep
    assert abs((y << (W + ex)) - ref[5]) << 53 > ref[5]
    y, ex = got[1]
    assert abs((y * 5 // 3 << (W + ex)) - ref[1]) << 53 > ref[1]


@pytest.mark.gpu
@pytest.mark.parametrize("K", [0, 1, 2, 4, 5, 6, 12, 13, 31, 32])
def test_device_against_model(K):
    """boys_eval gives the model's bits (cut to a double) where every step runs on
    the integer pipes (K < 6); from K = 6 on the first quarter of the steps runs in
    FP64, two roundings of 2^-53 a step, eight steps at most: 2^-48 relative."""
    import numpy as np
    import torch

    import paper_2512_10059_gb300 as pb
    pts = _points(K)
    got = pb.boys_eval(torch.tensor(pts, dtype=torch.float64, device="cuda:0"), K).cpu().numpy()
    for i, x in enumerate(pts):
        ref = _model(K, x)
        for l in range(K + 1):
            y, ex = ref[l]
            want = math.ldexp(y >> 10, ex + 10)
            if K < 6:
                assert got[l, i] == want, (K, l, x)
            else:
                assert abs(got[l, i] - want) <= 2.0 ** -48 * want, (K, l, x)
    assert np.all(np.isfinite(got))
