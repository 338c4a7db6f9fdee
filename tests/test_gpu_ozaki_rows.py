"""The folded density rows of the Ozaki analysis at the edges of their blocks: halves
of a row around multiples of 16 and 32 columns and around 146, where one accumulator
fill becomes two, odd and even counts (a middle cell, an odd half, rows that start off
16-byte boundaries), row counts around the 256-row tile, the longest rows taken, both
kinds of grid, and densities of mixed sign over many decades in one row, of scales next
to the ends of the float64 range, and zero, against the float64 CUDA-core path.

The bound: each cell enters with an error of at most 2^-49 of its row's scale, which is
up to 2^1.2 times the row's largest value, and so do the table's digits; over n_phi
cells of random sign that is 2^-47 sqrt(n_phi) <= 1.8e-13 of a row's largest term for
640, against moments that are sums of many rows: the bar of that comparison
elsewhere, 2e-13."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import gpu_solve, lib, phi_err, require_gpu

pytestmark = pytest.mark.gpu

CASES = [
    # polar, n_r, n_theta, n_phi, l_max
    (True, 3, 6, 1, 0), (True, 3, 6, 2, 1), (True, 3, 6, 31, 5), (True, 3, 6, 32, 5), (True, 3, 6, 33, 5), (True, 4, 8, 62, 7),
    (True, 4, 8, 63, 7), (True, 4, 8, 64, 7), (True, 4, 8, 65, 7), (True, 4, 8, 66, 7), (True, 32, 8, 96, 8), (True, 33, 8, 98, 8),
    (True, 2, 9, 290, 30), (True, 2, 9, 292, 31), (True, 2, 9, 293, 31), (True, 2, 9, 294, 31), (True, 2, 9, 320, 15), (True, 2, 9, 322, 15),
    (True, 2, 9, 383, 8), (True, 2, 9, 386, 9), (True, 2, 9, 639, 8), (True, 2, 9, 640, 16), (False, 3, 8, 34, 5), (False, 3, 8, 35, 5),
    (False, 9, 30, 90, 24), (False, 9, 30, 90, 33),
]


def build(case, scale):
    polar, n_r, n_theta, n_phi, lmax = case
    r = np.logspace(-2, 0, n_r + 1)
    spec = inputs.polar_grid(r, n_theta, n_phi, lmax) if polar else inputs.GridSpec("rows", r, n_theta, n_phi, 0.0, 0.0, lmax)
    rng = np.random.default_rng(5)
    rho = [(1.0 + rng.random((n_r, n_theta, n_phi))) * scale for _ in range(1 if polar else 2)]
    return spec, rho


def solve(g, rho, prec):
    if len(rho) == 2:
        return gpu_solve(g, rho[0], rho[1], gradient=False, prec=prec)
    import torch
    out = g.solve(torch.as_tensor(rho[0], device="cuda"), gradient=False, prec=prec)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


def compare(g, rho, scale=1.0):
    got, ref = solve(g, rho, "fp64_ozaki"), solve(g, rho, "fp64")
    for key in ref:   # over the scale, as their squares would leave the float64 range
        assert phi_err(got[key] / scale, ref[key] / scale) <= 2e-13, key


@pytest.mark.parametrize("case", CASES, ids=lambda c: ("polar" if c[0] else "yy") + "_" + "_".join(map(str, c[1:])))
def test_rows(case):
    require_gpu()
    yy = lib()
    spec, rho = build(case, 1.0)
    g = yy.Grid.from_spec(spec)
    g.prepare("fp64_ozaki")
    compare(g, rho)
    for x in rho:   # signs and decades within a row, and empty rows
        x *= np.where(np.arange(x.shape[2]) % 3 == 1, -1e-9, 1.0)
        x[:, 1] = 0.0
    compare(g, rho)
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    g.close()


@pytest.mark.parametrize("scale", [1e-290, 1e-271, 1e-270, 1e270, 1e272, 1e290])
@pytest.mark.parametrize("case", [(True, 4, 8, 64, 7), (True, 4, 8, 65, 7), (False, 4, 20, 60, 33)],
                         ids=lambda c: "_".join(map(str, c)))
def test_scales(case, scale):
    require_gpu()
    yy = lib()
    spec, rho = build(case, scale)
    g = yy.Grid.from_spec(spec)
    g.prepare("fp64_ozaki")
    compare(g, rho, scale)
    g.close()


@pytest.mark.parametrize("power", [-940, -880, 880, 940])
def test_scale_is_exact_across_the_far_rows(power):
    """rho 2^k gives 2^k times the result, bit for bit, also where rows are brought back
    by a power of two before their digits are taken (beyond 2^+-900)."""
    require_gpu()
    yy = lib()
    spec, rho = build((True, 4, 8, 65, 7), 1.0)
    g = yy.Grid.from_spec(spec)
    g.prepare("fp64_ozaki")
    one = solve(g, rho, "fp64_ozaki")
    far = solve(g, [np.ldexp(x, power) for x in rho], "fp64_ozaki")
    for key in one:
        assert np.array_equal(np.ldexp(one[key], power), far[key]), key
    g.close()
