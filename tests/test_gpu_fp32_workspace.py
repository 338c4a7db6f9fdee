"""YY_FP32 prepares the separable synthesis's tables and workspace only on grids that it serves.

At l_max 80 the trig table of 300 longitudes fits the synthesis's shared memory and that of 340
does not (there the dense contraction serves): the latter makes four allocations less, the
three transposed tables and the workspace of four fields."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, phi_err, require_gpu

pytestmark = pytest.mark.gpu


def allocations(yy, spec):
    for n in range(64):
        g = yy.Grid.from_spec(spec)
        yy.yy_debug_fail_alloc_after(n)
        st = yy.yy_grid_prepare(g.handle, yy.YY_FP32)
        yy.yy_debug_fail_alloc_after(-1)
        g.close()
        if st == yy.YY_OK:
            return n
    raise AssertionError("prepare never succeeds")


def test_only_where_it_serves():
    require_gpu()
    import torch
    yy = lib()
    specs = [inputs.polar_grid(np.array([0.1, 0.5, 1.0]), 2, n_phi, 80) for n_phi in (300, 340)]
    fits, dense = (allocations(yy, s) for s in specs)
    assert dense == fits - 4
    for spec in specs:
        g = yy.Grid.from_spec(spec)
        g.prepare("fp32")
        rho = torch.as_tensor(1.0 + np.random.default_rng(1).random((2, 2, spec.n_phi)), device="cuda")
        out = {p: g.solve(rho, prec=p)["phi"].cpu().numpy() for p in ("fp64", "fp32")}
        assert yy.yy_last_device_status(g.handle) == yy.YY_OK
        g.close()
        assert phi_err(out["fp32"], out["fp64"]) <= 1e-5
