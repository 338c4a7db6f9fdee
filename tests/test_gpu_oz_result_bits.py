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
