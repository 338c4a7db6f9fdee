"""The last step of the Ozaki synthesis: exact whole multiples of a row's unit to float64.

A row's unit is the last place in which any of its values differ from zero, 2^-50 of the
scales of its coefficients and of the trig table.  The multiples stay well below 2^53
here, so float64 holds them exactly, and about half of them are odd: of the hundreds of
rows some have an odd multiple in every column."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu

pytestmark = pytest.mark.gpu


def rows(g, rho):
    """Every row of every field of the polar grid's solve."""
    import torch
    out = g.solve(torch.as_tensor(rho, device="cuda"), gradient=True, prec="fp64_ozaki")
    torch.cuda.synchronize()
    return np.concatenate([out["phi"].cpu().numpy().reshape(-1, rho.shape[2]), out["grad"].cpu().numpy().reshape(-1, rho.shape[2])])


def last_places(v):
    """The exponent of each value's lowest bit (a large number for zero)."""
    m, e = np.frexp(v)
    whole = np.ldexp(m, 53).astype(np.int64)
    zeros = np.frexp((whole & -whole).astype(np.float64))[1] - 1
    return np.where(v == 0.0, 9999, e - 53 + zeros)


@pytest.mark.parametrize("n_phi, lmax", [(48, 20), (49, 31), (64, 32), (75, 35), (80, 63)])
def test_odd_multiples_in_every_column(n_phi, lmax):
    require_gpu()
    yy = lib()
    g = yy.Grid.from_spec(inputs.polar_grid(np.logspace(-1, 0, 10), 12, n_phi, lmax))
    g.prepare("fp64_ozaki")
    v = rows(g, 1.0 + np.random.default_rng(4).random((9, 12, n_phi)))
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    g.close()
    place = last_places(v)
    odd = place == place.min(axis=1, keepdims=True)
    assert odd.any(axis=0).all(), np.nonzero(~odd.any(axis=0))[0]


@pytest.mark.parametrize("lmax", [40, 63])
def test_single_units_at_the_bottom_of_the_range(lmax):
    """Rows whose unit is 2^-1023, below the normal range: a value of one unit stays one.

    A density that alternates along its rows excites the sine of order 32, whose derivative
    vanishes at the cells: g_phi is a few units there, of rounding alone (one row per shell, at
    the equator, so that neighbouring rows have about the same unit).  Rows are written 32
    at a time, by a quick form where all of them allow it.  The density is stepped by powers
    of two, so that the smallest unit of each group passes 2^-1023; at that step, and at
    those around it, some of these rows' values are a single unit."""
    require_gpu()
    yy = lib()
    g = yy.Grid.from_spec(inputs.polar_grid(np.logspace(-1, 0, 481), 1, 64, lmax))
    g.prepare("fp64_ozaki")
    rho = (1.0 - 2.0 * (np.arange(64) % 2)) * (1.0 + np.random.default_rng(6).random((480, 1, 1)))
    groups = lambda v: v[-480:].reshape(15, 32, 64)  # noqa: E731  (g_phi)
    least = last_places(groups(rows(g, rho))).min(axis=(1, 2))
    single = {at: 0 for at in range(-1025, -1020)}
    for power in range(-1026 - int(least.max()), -1019 - int(least.min())):
        v = groups(rows(g, np.ldexp(rho, power)))
        for at in single:
            single[at] += int((np.abs(v[least + power == at]) == 2.0 ** at).sum())
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    g.close()
    assert all(single[at] > 0 for at in single), single
