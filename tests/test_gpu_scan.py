"""The radial scan's coefficients at the edges of its register forms (2, 4, 8,
12, 18 and 24 radii per thread in 32 chunks, two passes above 768 zones), with
mode counts that leave the last block of four modes part empty, against the
radial sums of the moments in extended precision.

Every coefficient is a sum of at most n_r terms with factors <= 1 of the two
recurrences; float64 keeps it to a few ulp per step of the chunk chains and of
the five composition steps, and the two sums of opposite sign in g_r and the
ones at the centre are compared with the largest magnitude of their degree:
1e-13 covers 24 + 32 + 5 roundings of 1.1e-16 with a factor of ten.
"""

import math

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import gpu_solve, lib, require_gpu

pytestmark = pytest.mark.gpu


def _expected(r_edges, moments, lmax):
    """Phi, g_r and angular coefficients [3][n_r][n_lm] of one patch, G = 1."""
    ld = np.longdouble
    r = np.asarray(r_edges, dtype=ld)
    rm, rp = r[:-1], r[1:]
    n_r = rp.size
    out = np.zeros((3,) + moments.shape, dtype=ld)
    for l in range(lmax + 1):
        cols = slice(l * l, (l + 1) ** 2)
        A = moments[:, cols].astype(ld)
        c, d = np.zeros_like(A), np.zeros_like(A)
        x = np.zeros(A.shape[1], dtype=ld)
        for n in range(n_r):
            q = rm[n] / rp[n]
            x = q ** (l + 1) * x + rp[n] ** 2 * (1 - q ** (l + 3)) / (l + 3) * A[n]
            c[n] = x
        y = np.zeros(A.shape[1], dtype=ld)
        for n in range(n_r - 2, -1, -1):
            u = rp[n + 1] / rp[n]
            f = rp[n] ** 2 * (np.log(u) if l == 2 else (u ** (2 - l) - 1) / (2 - l))
            y = u ** (-l) * y + f * A[n + 1]
            d[n] = y
        k = 4 * math.pi / (2 * l + 1)
        out[0][:, cols] = -k * (c + d)
        out[1][:, cols] = -k * ((l + 1) * c - l * d) / rp[:, None]
        out[2][:, cols] = k * (c + d) / rp[:, None]
    return out


@pytest.mark.parametrize("n_r", [1, 31, 33, 64, 65, 128, 129, 256, 257, 384, 385, 576, 577, 768, 769])
@pytest.mark.parametrize("lmax,polar", [(0, False), (4, False), (5, True)])
def test_scan_coefficients(n_r, lmax, polar):
    require_gpu()
    yy = lib()
    r = np.logspace(-2, 0, n_r + 1)
    spec = inputs.polar_grid(r, 6, 12, lmax) if polar else inputs.GridSpec("scan", r, 6, 18, 0.0, 0.0, lmax)
    g = yy.Grid.from_spec(spec)
    rng = np.random.default_rng(n_r)
    rho = [rng.random((n_r, spec.n_theta, spec.n_phi)) for _ in range(1 if polar else 2)]
    if polar:
        import torch
        g.solve(torch.as_tensor(rho[0], device="cuda"))
        torch.cuda.synchronize()
    else:
        gpu_solve(g, rho[0], rho[1])
    patches = len(rho)
    n_lm = (lmax + 1) ** 2
    A = g.table(yy.YY_TABLE_MOMENTS_TOTAL).reshape(patches, n_r, n_lm)
    Q = g.table(yy.YY_TABLE_COEFF).reshape(3, patches, n_r, n_lm)
    for p in range(patches):
        ref = _expected(r, A[p], lmax)
        for f in range(3):
            for l in range(lmax + 1):
                cols = slice(l * l, (l + 1) ** 2)
                scale = np.abs(ref[f][:, cols]).max()
                err = np.abs(Q[f, p][:, cols] - ref[f][:, cols]).max()
                assert err <= 1e-13 * scale, (p, f, l, float(err / scale) if scale else float(err))
    g.close()
