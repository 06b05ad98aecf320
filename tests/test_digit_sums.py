"""The exact sums of the kernels' digit epilogues, emulated in float32 on the CPU.

The target projection adds its levels L_l 2^(-8 l) (integers, |L_l| <= 2^23)
by three operations each, v' = v + x, r = x - (v' - v) (Fast2Sum).  That is
exact when v is an integer multiple of the last place of x, whatever their
order of magnitude: checked here against integers, at the bounds and for
cancelling and tiny leading sums.  The sweep product adds its groups in
double-float by the same means.
"""
from fractions import Fraction

import numpy as np
import pytest

F = np.float32


def _fma(x, f, v):
    # x f is exact in float64 for a float32 x and a power of two f; the sum
    # has at most 24 + 40 bits between its ends and is rounded once more to
    # float32 only where float64 holds it exactly (asserted by the caller)
    return F(np.float64(x) * f + np.float64(v))


def fast2sum(v, x, f):
    v2 = _fma(x, f, v)
    return v2, _fma(x, f, F(v - v2))


@pytest.mark.parametrize("base", [8])
@pytest.mark.parametrize("lead", [0, 1, 255, 1 << 14, 1 << 21])
def test_level_sums_are_exact(base, lead):
    rng = np.random.default_rng(base + lead)
    n, bound = 4000, 1 << 23
    L = [np.clip(rng.integers(-lead, lead + 1, n), -bound, bound)]
    L += [rng.integers(-bound, bound + 1, n) for _ in range(3)]
    L[1][:8] = [bound, -bound, 1, -1, 0, bound - 1, 1 - bound, 2]
    L[2][4:8] = [bound, -bound, bound, -bound]
    v = F(L[0])
    total = L[0].astype(object)
    rest = [0] * n
    for t in range(1, 4):
        v, r = fast2sum(v, F(L[t]), 2.0 ** (-base * t))
        total = total * (1 << base) + L[t]
        rest = [a * (1 << base) + int(np.float64(b) * 2.0 ** (base * t + 8)) for a, b in zip(rest, r)]
        have = [int(np.float64(a) * 2.0 ** (base * t + 8)) + b for a, b in zip(v, rest)]
        assert have == [int(x) << 8 for x in total]


def _fma2(x, y, z):
    # 48-bit product and a sum in at least 64 bits, then rounded to float32
    return (x.astype(np.longdouble) * y.astype(np.longdouble) + z.astype(np.longdouble)).astype(F)


@pytest.mark.parametrize("spread", [0, 8])     # orders of magnitude among the scales
@pytest.mark.parametrize("lead", [0, 1, 20, 24])
@pytest.mark.parametrize("groups", [1, 5, 86])
def test_sweep_product_sum(groups, lead, spread):
    """The sweep product's epilogue: per group D_0 + D_1 2^-10 as an exact pair,
    times the scale, added by a two-sum of the rounded product whose last
    difference takes the unrounded one.  Only the low part is rounded: at most
    four times on the way to a group's term and once per addition, by 2^-24 of
    what is rounded each time."""
    rng = np.random.default_rng(100 * groups + lead + spread)
    n, bound = 300, 128 * 255 * 512
    c10, c20 = np.full(n, 2.0 ** -10, F), np.full(n, 2.0 ** -20, F)
    H, L, low = np.zeros(n, F), np.zeros(n, F), np.zeros(n)
    exact = np.zeros(n, dtype=object) + Fraction(0)
    for _ in range(groups):
        s = F(rng.uniform(0.5, 2, n) * 2.0 ** rng.integers(-spread, spread + 1, n))
        D = [rng.integers(-min(bound, 2 ** lead - 1), min(bound, 2 ** lead - 1) + 1, n)]
        D += [rng.integers(-bound, bound + 1, n) for _ in range(3)]
        D[1][:3] = [bound, -bound, 0]
        d0, d1, d2, d3 = (F(x) for x in D)
        vh = _fma2(d1, c10, d0)
        split = _fma2(d1, c10, d0 - vh)
        assert np.array_equal(vh.astype(float) + split, D[0] + D[1] * 2.0 ** -10)    # exact
        vl = _fma2(_fma2(d3, c10, d2), c20, split)
        sm = H + vh * s
        nb = H - sm
        er = (H - (sm + nb)) + _fma2(vh, s, nb)
        low += np.abs(vl.astype(float) * s) + np.abs(H - (sm + nb)) + np.abs(_fma2(vh, s, nb))
        H, L = sm, L + _fma2(vl, s, er)
        exact += [Fraction(float(a)) * (Fraction(int(x)) + Fraction(int(y), 1 << 10) + Fraction(int(z), 1 << 20)
                                        + Fraction(int(w), 1 << 30)) for a, x, y, z, w in zip(s, *D)]
    err = [abs(Fraction(float(h)) + Fraction(float(l)) - e) for h, l, e in zip(H, L, exact)]
    assert all(float(e) <= (groups + 4) * 2.0 ** -24 * b for e, b in zip(err, low))


def test_float32_widened_by_integer_operations():
    """float32 -> float64 by re-biasing the exponent: exact for zeros and all
    normal numbers (the kernels convert the others)."""
    rng = np.random.default_rng(3)
    b = np.concatenate([rng.integers(0, 1 << 32, 200000, dtype=np.uint64),
                        [0, 1 << 31, 0x00800000, 0x007FFFFF, 1, 0x7F7FFFFF, 0xFF7FFFFF, 0x80800000, 0x7F800000]])
    b = b.astype(np.uint32)
    m = b & np.uint32(0x7FFFFFFF)
    rare = (m - np.uint32(1) < 0x007FFFFF) | (m >= 0x7F800000)
    x = b.view(F)
    assert np.array_equal(rare, ~(np.isfinite(x) & ((x == 0) | (np.abs(x) >= np.finfo(F).tiny))))
    hi = np.where(m > 0, (m >> np.uint32(3)) + np.uint32(896 << 20), 0).astype(np.uint64)
    hi |= (b & np.uint32(1 << 31)).astype(np.uint64)
    lo = ((m.astype(np.uint64) << np.uint64(29)) & np.uint64(0xFFFFFFFF))
    bits = ((hi << np.uint64(32)) | lo)[~rare]
    assert np.array_equal(bits, x[~rare].astype(np.float64).view(np.uint64))
