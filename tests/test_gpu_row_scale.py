"""Every density row of the Ozaki analysis enters with 48 bits of its largest value.

Densities constant over each row of a polar grid (weights of 1), each 48 bits long
with mantissas from 1.84 to 2, where the sum of the operands' upper words overstates
the product's exponent, or from 1 to 2, and the same with one added in the 48th bit.  That bit
is zero before, so a row cut to 47 bits would round both to the same digits (ties
to even), and the same digits give the same moments in every bit.  How far a moment
moves says little, as the polar stage rounds to about that bit; of a shell's ten
rows and six axisymmetric moments some move."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_phi", [16, 17])
@pytest.mark.parametrize("power", [0, -950])
@pytest.mark.parametrize("least", [1.0, 1.84])
def test_the_48th_bit_enters(n_phi, power, least):
    require_gpu()
    import torch
    yy = lib()
    n_r, n_theta = 32, 10
    spec = inputs.polar_grid(np.logspace(-1, 0, n_r + 1), n_theta, n_phi, 5)
    g = yy.Grid.from_spec(spec)
    g.prepare("fp64_ozaki")
    rng = np.random.default_rng(3)
    X = rng.integers(int(least * 2 ** 46), 2 ** 47 - 8, (n_r, n_theta, 1)) // 4 * 4
    moments = []
    for bit in (0, 1):
        rho = np.ldexp((X + bit).astype(np.float64), power - 46) * np.ones(n_phi)
        g.solve(torch.as_tensor(rho, device="cuda"), prec="fp64_ozaki")
        torch.cuda.synchronize()
        moments.append(g.table(yy.YY_TABLE_MOMENTS).reshape(n_r, -1))
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    g.close()
    same = np.all(moments[0] == moments[1], axis=1)
    assert not same.any(), np.nonzero(same)[0]
