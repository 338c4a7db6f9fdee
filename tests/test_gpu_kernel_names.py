"""Which kernels a solve runs, by the names that a profiled solve reports: the grids at the
edges of the folds, the digit rows and the streamed packing take the kernels that their tests are
about, and those past an edge the others."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu
from tests.test_gpu_folds import GRIDS as FOLDS
from tests.test_gpu_folds import _spec as fold_spec
from tests.test_gpu_ozaki_rows import CASES as ROWS
from tests.test_gpu_stream_pieces import SIZES as PIECES

pytestmark = pytest.mark.gpu


def kernels(spec, prec, method="auto"):
    """Names of the kernels of a profiled solve of Phi and the gradient."""
    import torch
    yy = lib()
    g = yy.Grid.from_spec(spec)
    g.prepare(prec)
    g.set_analysis(method)
    rho = [torch.ones((spec.n_r, spec.n_theta, spec.n_phi), dtype=torch.float64, device="cuda") for _ in range(1 if spec.polar else 2)]
    yy.yy_grid_set_profiling(g.handle, 1)
    g.solve(*rho, gradient=True, prec=prec)
    torch.cuda.synchronize()
    names = {n for n, _ in yy.yy_grid_kernels_ms(g.handle)}
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    g.close()
    return names


def test_folds():
    require_gpu()
    for case in FOLDS:
        assert {"k_sep_phi64", "k_sep_theta64", "k_synth_f64"} <= kernels(fold_spec(*case), "fp64"), case
        assert {"k_sep_phi32", "k_sep_theta32", "k_theta32", "k_phi32"} <= kernels(fold_spec(*case), "fp32"), case
        assert not any("sep" in n or n == "k_synth_f64" for n in kernels(fold_spec(*case), "fp64", "dense")), case


def test_digit_rows():
    require_gpu()
    r = np.logspace(-2, 0, 4)
    for polar, _, n_theta, n_phi, lmax in ROWS:
        spec = inputs.polar_grid(r, n_theta, n_phi, lmax) if polar else inputs.GridSpec("rows", r, n_theta, n_phi, 0.0, 0.0, lmax)
        assert {"k_rhow_ozaki", "k_oz_analysis", "k_sep_theta_ff", "k_q_ff", "k_theta_ff", "k_oz_synth"} <= kernels(spec, "fp64_ozaki"), (n_theta, n_phi, lmax)
    assert {"k_sep_phi64", "k_oz_synth"} <= kernels(inputs.polar_grid(r, 6, 641, 8), "fp64_ozaki")   # rows too long for the digits


@pytest.mark.parametrize("prec", ["fp16x2", "bf16x3"])
def test_packed_rows(prec):
    require_gpu()
    grid = lambda n_theta, n_phi: inputs.GridSpec("pieces", np.linspace(0.0, 1.0, 4), n_theta, n_phi, 0.0, 0.0, 4)  # noqa: E731
    for size in PIECES:
        assert "k_pack_stream" in kernels(grid(*size), prec), size
    for size in ((63, 131), (32, 64), (129, 192)):   # an odd length, a short row, more than three pieces
        names = kernels(grid(*size), prec)
        assert "k_pack_stream" not in names and "k_pack_reg/densities" in names, size
