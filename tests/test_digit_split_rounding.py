"""The base-1024 digit split of the Ozaki synthesis (ff_digits_x2) in binary32
arithmetic: every step as the kernel does it, a fused multiply-add as the exact
product and sum rounded once.  The digits have to stay within the bounds that
the level sums and fp16 need, and to give the value to half a unit of the last
digit plus what the third digit's remainder rounds off (2^-25 of its unit,
2^-55 of the scale)."""

from fractions import Fraction

import numpy as np
import pytest

f32 = np.float32
M = f32(1.5 * 2 ** 23)


def fma(a, b, c):
    """round-to-nearest-even binary32 of a b + c, exact before the rounding"""
    x = Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c))
    if x == 0:
        return f32(0.0)
    y = f32(float(x))                        # nearest up to double rounding: corrected below
    best = min((y, np.nextafter(y, f32(np.inf)), np.nextafter(y, f32(-np.inf))),
               key=lambda v: (abs(Fraction(float(v)) - x), int(np.array(v).view(np.uint32)) & 1))
    return f32(best)


def digits(hi, lo, K):
    p1, p2 = f32(2.0 ** (K >> 1)), f32(2.0 ** (K - (K >> 1)))
    H = f32(f32(hi * p1) * p2)
    L = f32(f32(f32(lo * p1) * p2) * f32(2 ** 20))
    k = f32(1024)
    d0 = f32(f32(H + M) - M)
    r0 = f32(H - d0)
    d1 = f32(fma(r0, k, M) - M)
    r1 = fma(r0, k, f32(-d1))
    d2 = f32(f32(fma(r1, k, L) + M) - M)
    r2 = f32(fma(r1, k, f32(-d2)) + L)
    d3 = f32(fma(r2, k, M) - M)
    r3 = fma(r2, k, f32(-d3))
    d4 = f32(fma(r3, k, M) - M)
    return [d0, d1, d2, d3, d4]


def _pairs(rng, n, e):
    """float-float values below 2^(e - 1), many of them far below the scale"""
    x = (rng.random(n) - 0.5) * 2.0 ** e * 2.0 ** -rng.integers(0, 45, n)
    x[:4] = [2.0 ** (e - 1) * (1 - 2.0 ** -24), -2.0 ** (e - 1) * (1 - 2.0 ** -24), 2.0 ** (e - 11), 0.0]
    hi = x.astype(f32)
    half_ulp = np.spacing(np.abs(hi)) / 2
    lo = (half_ulp * (2 * rng.random(n) - 1)).astype(f32)
    lo[4:8] = half_ulp[4:8]
    return hi, np.where(hi == 0, f32(0), lo)


@pytest.mark.parametrize("e", [-60, 0, 3, 70])
def test_digits_give_the_value(e):
    rng = np.random.default_rng(e + 100)
    for hi, lo in zip(*_pairs(rng, 300, e)):
        d = [int(v) for v in digits(hi, lo, 10 - e)]
        assert all(abs(v) <= (528 if s == 2 else 512) for s, v in enumerate(d)), d
        exact = (Fraction(float(hi)) + Fraction(float(lo))) / Fraction(2) ** e
        got = sum(Fraction(v, 1024 ** (s + 1)) for s, v in enumerate(d))
        assert abs(got - exact) <= Fraction(1, 2 ** 51) + Fraction(1, 2 ** 54), (float(hi), float(lo), d)
