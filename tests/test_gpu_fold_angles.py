"""The float64 folds use one trig value for up to eight cells: it is that of all of these cells.

The angle at which the solve evaluated each column, from Phi and the solve's own coefficients: Phi in
extended precision at (k - (n_phi - 1) / 2) cells of (3 pi / 2 + 2 delta_phi) / n_phi, and the shift of the angle that
explains the solve's differences from it, by least squares over the rows of one shell.  The shift is zero but
for the roundings: a term of order m takes some (l_max - m) / 2 + l_max / 2 additions and a dozen roundings
of table values and products, each up to 2^-53 of its size and evenly spread, which gives the
shift a standard deviation; six of them are allowed.  (An angle rounded at the size of pi is off by up to eight
times 2^-53, some twenty of them.)"""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288419716939937510582097494459")


@pytest.mark.parametrize("n_theta, n_phi, buffer, lmax, m0", [(40, 48, 2, 40, 36), (39, 47, 1, 40, 35), (40, 46, 0, 30, 29),
                                                                (40, 60, 0, 40, 36), (39, 45, 0, 40, 38)])
def test_angles(n_theta, n_phi, buffer, lmax, m0):
    require_gpu()
    import torch
    yy = lib()
    n_r, n_lm = 1, (lmax + 1) ** 2
    b = buffer * 1.5 * np.pi / (n_phi - 2 * buffer)
    g = yy.Grid.from_spec(inputs.GridSpec("angles", np.linspace(0.5, 1.0, n_r + 1), n_theta, n_phi, 0.1, b, lmax))
    phi = (np.arange(n_phi) - LD(n_phi - 1) / 2) * (3 * PI / 2 + 2 * LD(b)) / n_phi
    rho = np.cos(m0 * phi + LD(0.7)).astype(np.float64) * np.ones((n_r, n_theta, 1))
    out = g.solve(torch.as_tensor(rho, device="cuda"), torch.zeros((n_r, n_theta, n_phi), dtype=torch.float64, device="cuda"), prec="fp64")
    torch.cuda.synchronize()
    got = out["phi_yin"].cpu().numpy().astype(LD)
    Q = g.table(yy.YY_TABLE_COEFF).reshape(3, 2, n_r, n_lm)[0, 0].astype(LD)
    Y = g.table(yy.YY_TABLE_SYNTH).reshape(n_theta, n_phi, n_lm).astype(LD)
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    g.close()
    half = (n_theta + 1) // 2   # rows whose own polar factors serve (sqrt(cos^2 + sin^2) of the modes' pairs)
    ref, slope, var = (np.zeros((n_r, half, n_phi), LD) for _ in range(3))
    for l in range(lmax + 1):
        ref += Q[:, l * l, None, None] * Y[None, :half, :1, l * l]
        for m in range(1, l + 1):
            i, c, s = l * l + 2 * m - 1, np.cos(m * phi), np.sin(m * phi)
            P = np.sqrt(Y[:half, 0, i] ** 2 + Y[:half, 0, i + 1] ** 2) * np.sign(Y[:half, 0, i] * c[0] + Y[:half, 0, i + 1] * s[0])
            a, d = (Q[:, at, None, None] * P[None, :, None] for at in (i, i + 1))
            ref += a * c + d * s
            slope += m * (d * c - a * s)
            var += ((a * c) ** 2 + (d * s) ** 2) * ((lmax - m) / 2 + lmax / 2 + 12) * 2.0 ** -106 / 3
    norm = (slope ** 2).sum((0, 1))
    shift = ((got[:, :half] - ref) * slope).sum((0, 1)) / norm
    spread = np.sqrt((slope ** 2 * var).sum((0, 1))) / norm
    sigmas = np.abs(shift / spread).astype(np.float64)
    assert sigmas.max() <= 6.0, (sigmas.max(), float(np.abs(shift).max() * 2.0 ** 53))
