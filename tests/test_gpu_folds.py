"""The CUDA-core separable stages on grids at the edges of their tiles and folds.

The float64 stages fold the cells by their symmetries (theta about the equator,
phi about the mirror axis, and phi -> pi - phi where pi is a whole number of
cells); the fp32 stages take tiles of rows and longitudes.  Each grid is solved
in separable and in dense form: both are float64 (or fp32) evaluations of the
same sums, so they agree to the forms' bars against the oracle (1e-13, and 1e-6
between float64 and the separable fp32 form).
"""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import grad_err, gpu_solve, lib, phi_err, require_gpu

pytestmark = pytest.mark.gpu

# (polar, n_r, n_theta, n_phi, buffer cells, l_max): pi a whole number of cells for
# n_phi - 2 buffer a multiple of 3 (Yin-Yang) or n_phi even (polar); odd and even
# rows and columns; one row, one column, one shell; more rows than one tile, fewer
# than one; an odd and an even distance between a column and its partner
GRIDS = [
    (False, 5, 9, 27, 0, 6), (False, 5, 10, 30, 0, 7), (False, 3, 8, 25, 0, 5), (False, 4, 7, 26, 0, 6),
    (False, 6, 12, 34, 2, 8), (False, 2, 11, 31, 1, 9), (False, 40, 17, 41, 0, 13), (False, 1, 1, 3, 0, 1),
    (False, 1, 2, 1, 0, 0), (False, 33, 45, 135, 0, 15), (False, 3, 30, 90, 0, 33), (False, 2, 40, 120, 0, 64),
    (True, 7, 8, 16, 0, 5), (True, 7, 9, 18, 0, 6), (True, 3, 9, 17, 0, 6), (True, 1, 4, 2, 0, 2), (True, 50, 32, 60, 0, 20),
]


def _spec(polar, n_r, n_theta, n_phi, b, lmax):
    r = np.logspace(-2, 0, n_r + 1)
    if polar:
        return inputs.polar_grid(r, n_theta, n_phi, lmax)
    return inputs.GridSpec("fold", r, n_theta, n_phi, b * 0.5 * np.pi / max(1, n_theta - 2 * b),
                           b * 1.5 * np.pi / max(1, n_phi - 2 * b), lmax)


def _rho(spec, seed):
    rng = np.random.default_rng(seed)
    shape = (spec.n_r, spec.n_theta, spec.n_phi)
    r = 0.5 * (spec.r_edges[:-1] + spec.r_edges[1:])[:, None, None]
    return [np.exp(-3 * r) * (1 + 0.3 * rng.random(shape)) for _ in range(1 if spec.polar else 2)]


@pytest.mark.parametrize("case", GRIDS, ids=lambda c: ("polar" if c[0] else "yy") + "_" + "_".join(map(str, c[1:])))
@pytest.mark.parametrize("gradient", [False, True])
def test_separable_matches_dense(case, gradient):
    require_gpu()
    yy = lib()
    spec = _spec(*case)
    rho = _rho(spec, 7)
    rho += [None] * (2 - len(rho))

    def solve(prec, method):
        g = yy.Grid.from_spec(spec)
        g.prepare(prec)
        g.set_analysis(method)
        if spec.polar:
            import torch
            x = torch.as_tensor(rho[0], device="cuda")
            out = g.solve(x, gradient=gradient, prec=prec)
            torch.cuda.synchronize()
            out = {k: v.cpu().numpy() for k, v in out.items()}
        else:
            out = gpu_solve(g, rho[0], rho[1], gradient=gradient, prec=prec)
        assert yy.yy_last_device_status(g.handle) == yy.YY_OK
        g.close()
        return out

    dense = solve("fp64", "dense")
    for prec, tol in (("fp64", 1e-13), ("fp32", 1e-6)):
        got = solve(prec, "auto")
        assert got.keys() == dense.keys()
        for key in dense:
            if key.startswith("phi"):
                assert phi_err(got[key], dense[key]) <= tol, (prec, key)
            elif np.any(dense[key]):
                assert grad_err(got[key], dense[key]) <= tol, (prec, key)
