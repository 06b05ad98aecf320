"""The exact sums of the kernels' digit epilogues, emulated in float32 on the CPU.

The target projection adds its levels L_l 2^(-8 l) (integers, |L_l| <= 2^23)
by three operations each, v' = v + x, r = x - (v' - v) (Fast2Sum).  That is
exact when v is an integer multiple of the last place of x, whatever their
order of magnitude: checked here against integers, at the bounds and for
cancelling and tiny leading sums.
"""
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
