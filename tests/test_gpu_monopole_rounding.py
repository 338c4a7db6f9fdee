"""The float64 synthesis adds the monopole last.

On a nearly spherical density the monopole is almost the whole of Phi and g_r.
It is added last in both sums (over l, then over the slots), so each value takes
two roundings at its own size, 2^-53 each.  Everything else is rounded at the
size of the other terms: of the order of their number (chains of 2 l_max + 1
and l_max + 1 terms) and of l_max radians times the rounding of an angle, below
8 pi l_max + 3 (2 l_max + 1) units of 2^-53 of the sum of their magnitudes.
Against the same coefficients and table evaluated in extended precision.
"""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu

pytestmark = pytest.mark.gpu

# (polar, n_theta, n_phi, l_max): pi / 2 a whole number of cells, pi alone, neither; odd rows and columns; odd and even degree
GRIDS = [(False, 12, 36, 8), (False, 13, 34, 7), (True, 9, 18, 7), (True, 8, 16, 6), (True, 9, 17, 5)]
U = 2.0 ** -53


@pytest.mark.parametrize("case", GRIDS, ids=lambda c: ("polar" if c[0] else "yy") + "_" + "_".join(map(str, c[1:])))
def test_two_roundings_of_the_monopole(case):
    require_gpu()
    import torch
    yy = lib()
    polar, n_theta, n_phi, lmax = case
    n_r, n_lm = 40, (lmax + 1) ** 2
    r = np.logspace(-2, 0, n_r + 1)
    spec = inputs.polar_grid(r, n_theta, n_phi, lmax) if polar else inputs.GridSpec("mono", r, n_theta, n_phi, 0.0, 0.0, lmax)
    rng = np.random.default_rng(11)
    mid = 0.5 * (r[:-1] + r[1:])[:, None, None]
    rho = [torch.as_tensor(np.exp(-3 * mid) * (1 + 1e-4 * rng.random((n_r, n_theta, n_phi))), device="cuda")
           for _ in range(1 if polar else 2)]
    g = yy.Grid.from_spec(spec)
    out = g.solve(*(rho if not polar else rho + [None]), gradient=True, prec="fp64")
    torch.cuda.synchronize()
    out = {k: v.cpu().numpy() for k, v in out.items()}
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    names = [("phi", "grad")] if polar else [("phi_yin", "grad_yin"), ("phi_yang", "grad_yang")]
    Q = g.table(yy.YY_TABLE_COEFF).reshape(3, len(names), n_r, n_lm).astype(np.longdouble)
    Y = g.table(yy.YY_TABLE_SYNTH).reshape(-1, n_lm).astype(np.longdouble)
    g.close()
    per_term = 8 * np.pi * lmax + 3 * (2 * lmax + 1)
    for p, (phi, grad) in enumerate(names):
        for what, coef, got in (("phi", Q[0, p], out[phi]), ("g_r", Q[1, p], out[grad][0])):
            ref = coef @ Y.T
            others = np.abs(coef[:, 1:]) @ np.abs(Y[:, 1:].T)
            large = np.abs(coef[:, :1] @ Y[:, :1].T)
            err = np.abs(got.reshape(n_r, -1).astype(np.longdouble) - ref)
            bound = U * (np.abs(ref) + large + per_term * others)
            assert float((err / bound).max()) <= 1.0, (phi, what, float((err / (U * np.abs(ref))).max()))
