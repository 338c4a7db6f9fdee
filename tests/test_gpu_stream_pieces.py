"""Long density rows packed piece by piece (8192 values each): row lengths at the edges
of one, two and three pieces, more rows than SMs, so that blocks start the next row's
pieces while they hold this one, against the float64 path at the bars of the
tensor-core forms against it (1e-6 for the potential)."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import gpu_solve, lib, phi_err, require_gpu

pytestmark = pytest.mark.gpu

# n_theta x n_phi = 8190, 8192, 8194, 16380, 16384, 16390, 24576 values
SIZES = [(63, 130), (64, 128), (34, 241), (90, 182), (128, 128), (110, 149), (128, 192)]


@pytest.mark.parametrize("size", SIZES, ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("prec", ["fp16x2", "bf16x3"])
def test_pieces(size, prec):
    require_gpu()
    yy = lib()
    n_r = 170
    r = np.linspace(0.0, 1.0, n_r + 1)
    spec = inputs.GridSpec("pieces", r, size[0], size[1], 0.0, 0.0, 4)
    rng = np.random.default_rng(3)
    # rows of very different levels: a piece of another row would show
    level = 10.0 ** rng.uniform(-2, 2, (n_r, 1, 1))
    rho = [level * (1.0 + 0.5 * rng.random((n_r,) + size)) for _ in range(2)]
    g = yy.Grid.from_spec(spec)
    g.prepare(prec)
    got, ref = gpu_solve(g, rho[0], rho[1], prec=prec), gpu_solve(g, rho[0], rho[1], prec="fp64")
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    for key in ref:
        assert phi_err(got[key], ref[key]) <= 1e-6, key
    g.close()
