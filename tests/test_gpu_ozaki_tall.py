"""YY_FP64_OZAKI on grids of many polar rows at l_max 63: past the shared memory of the
float-float polar stage (the float64 stage serves) and, from 227 rows, past that of the
float64 stage too (the dense float64 analysis serves), against the float64 path: the bar
of that comparison elsewhere, 2e-13."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, phi_err, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_theta", [98, 100, 226, 227, 230])
def test_against_float64(n_theta):
    require_gpu()
    import torch
    yy = lib()
    g = yy.Grid.from_spec(inputs.polar_grid(np.array([0.1, 0.5, 1.0]), n_theta, 64, 63))
    g.prepare("fp64_ozaki")
    rho = torch.as_tensor(1.0 + np.random.default_rng(9).random((2, n_theta, 64)), device="cuda")
    out = {p: g.solve(rho, prec=p)["phi"].cpu().numpy() for p in ("fp64", "fp64_ozaki")}
    assert yy.yy_last_device_status(g.handle) == yy.YY_OK
    g.close()
    assert phi_err(out["fp64_ozaki"], out["fp64"]) <= 2e-13
