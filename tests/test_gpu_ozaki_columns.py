"""The folded columns of the Ozaki synthesis at the edges of its tiles: longitude
counts around multiples of twice the 48-column tile, odd and even (a cell that is
its own mirror, rows that start off 16-byte boundaries, a first folded cell of
either parity), both slot layouts (l_max up to 31 and above), row counts around
the 256-row cell tile, with and without the gradient, against the float64
CUDA-core path (the bar of that comparison elsewhere: 2e-13)."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import grad_err, gpu_solve, lib, phi_err, require_gpu

pytestmark = pytest.mark.gpu

CASES = [
    # polar, n_r, n_theta, n_phi, l_max
    (False, 3, 8, 3, 1), (False, 4, 9, 26, 5), (False, 4, 9, 27, 5), (False, 4, 9, 28, 5), (False, 16, 8, 94, 9),
    (False, 16, 8, 95, 9), (False, 17, 8, 96, 9), (False, 9, 12, 97, 9), (False, 9, 12, 98, 9), (False, 5, 20, 192, 31),
    (False, 5, 20, 193, 32), (False, 5, 22, 66, 33), (False, 3, 40, 110, 63), (True, 4, 10, 1, 0), (True, 4, 10, 2, 1), (True, 5, 13, 33, 8), (True, 6, 12, 96, 8),
    (True, 6, 12, 98, 8), (True, 3, 40, 191, 35),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: ("polar" if c[0] else "yy") + "_" + "_".join(map(str, c[1:])))
@pytest.mark.parametrize("gradient", [False, True])
def test_ozaki_columns(case, gradient):
    require_gpu()
    yy = lib()
    polar, n_r, n_theta, n_phi, lmax = case
    r = np.logspace(-2, 0, n_r + 1)
    spec = inputs.polar_grid(r, n_theta, n_phi, lmax) if polar else inputs.GridSpec("cols", r, n_theta, n_phi, 0.0, 0.0, lmax)
    rng = np.random.default_rng(11)
    rho = [1.0 + 0.5 * rng.random((n_r, n_theta, n_phi)) for _ in range(1 if polar else 2)]
    g = yy.Grid.from_spec(spec)
    g.prepare("fp64_ozaki")

    def solve(prec):
        if not polar:
            return gpu_solve(g, rho[0], rho[1], gradient=gradient, prec=prec)
        import torch
        out = g.solve(torch.as_tensor(rho[0], device="cuda"), gradient=gradient, prec=prec)
        torch.cuda.synchronize()
        return {k: v.cpu().numpy() for k, v in out.items()}

    got, ref = solve("fp64_ozaki"), solve("fp64")
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    for key in ref:
        if key.startswith("phi"):
            assert phi_err(got[key], ref[key]) <= 2e-13, key
        else:
            assert grad_err(got[key], ref[key]) <= 2e-13, key
    g.close()
