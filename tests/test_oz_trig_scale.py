"""The scale of the Ozaki synthesis's trig digits: the first one under which every level
sum is exact, and none where no scale is (instead of digits whose sums would round).

Exact: 528 times the sum of the three top base-1024 digits' magnitudes over the 32 slots
of a class stays below 2^24, an average of 993 per slot."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import build, yy


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def bad(q, top):
    """A value whose digits under 2^-q are top, 512, 512, 0, 0."""
    return 2.0 ** q * (top / 2.0 ** 10 + 512 / 2.0 ** 20 + 512 / 2.0 ** 30)


def table(lmax, n_phi):
    ph = -0.75 * np.pi + 1.5 * np.pi / n_phi * (np.arange(n_phi) + 0.5)
    rows = [np.ones(n_phi)]
    for m in range(1, lmax + 1):
        rows += [np.cos(m * ph), np.sin(m * ph)]
    return np.array(rows)


@pytest.mark.parametrize("lmax, n_phi", [(0, 3), (8, 48), (25, 270), (31, 77), (40, 185), (63, 24), (63, 639)])
def test_trig_tables_take_a_quarter(lmax, n_phi):
    assert yy.yy_debug_oz_trig_scale(table(lmax, n_phi)) == 2


@pytest.mark.parametrize("lmax", [31, 63])
def test_the_next_scale_and_none(lmax):
    t = table(lmax, 24)
    t[1:, 5] = bad(2, 250)      # 1274 a slot under 2^-2
    assert yy.yy_debug_oz_trig_scale(t) == 3
    t[1:, 7] = -bad(3, 120)     # 1144 under 2^-3
    assert yy.yy_debug_oz_trig_scale(t) == 4
    t[1:, 11] = bad(4, 60)      # 1084 under 2^-4
    assert yy.yy_debug_oz_trig_scale(t) == -1


def test_invalid_arguments():
    assert yy.yy_debug_oz_trig_scale(np.ones((129, 2))) == -2
