"""The scale of a digit row from the operands' upper words (k_rhow_ozaki): the exponent
and mantissa bits of a positive float64, read as one number, are its logarithm less at
most 0.0861, so (hi(rho) + hi(w) + 180700) >> 20 bounds the product's exponent: every
|rho w| is below 2^(e - 1) and, since the two shortfalls and the margin together stay below
1.35 bits, the largest is above 2^(e - 1 - 1.35)."""

import numpy as np


def hi(v):
    return (v.view(np.uint64) >> np.uint64(32)) & np.uint64(0x7FFFFFFF)


def check(x, w):
    e = ((hi(x) + hi(w) + np.uint64(180700)) >> np.uint64(20)).astype(np.int64) - 2044
    m, ex = np.frexp(x * w)
    r = np.ldexp(m, (ex - (e - 1)).astype(np.int64))
    assert r.max() < 1.0 and r.min() > 2.0 ** -1.35


def test_scale_bounds_every_product():
    rng = np.random.default_rng(2)
    for _ in range(20):
        n = 100000
        check(np.ldexp(1 + rng.random(n), rng.integers(-300, 300, n)), np.ldexp(1 + rng.random(n), rng.integers(-300, 1, n)))


def test_scale_at_the_worst_mantissas():
    # 2^0.5287 has the largest shortfall; the ends of the mantissa; low words that are not seen
    m = np.concatenate([1 + np.linspace(0, 1, 4097)[:-1], np.nextafter(1 + np.linspace(0, 1, 4097)[1:], 0), [1.0, np.nextafter(2.0, 0)]])
    for e in (-1, 0, 7):
        x = np.ldexp(m, e)
        for w in (1.0, 1 / np.log(2), np.nextafter(1.0, 0), 0.5 / np.log(2)):
            check(x, np.full_like(x, w))
