"""yy_grid_prepare(YY_FP32) with an allocation that fails: all of its tables or none.

Whichever allocation fails, the form stays unprepared (a solve is refused), and the next
prepare completes it: the results are those of a grid prepared at once, bit for bit."""

import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu

pytestmark = pytest.mark.gpu


def prepared_after(yy, spec, n):
    """A grid whose prepare met a failure at the n-th allocation, and what it returned."""
    g = yy.Grid.from_spec(spec)
    yy.yy_debug_fail_alloc_after(n)
    st = yy.yy_grid_prepare(g.handle, yy.YY_FP32)
    yy.yy_debug_fail_alloc_after(-1)
    return g, st


def test_every_allocation():
    require_gpu()
    import torch
    yy = lib()
    spec = inputs.tiny_grid()
    rho = [torch.as_tensor(x, device="cuda") for x in inputs.density_for(spec)]
    g = yy.Grid.from_spec(spec)
    g.prepare("fp32")
    ref = g.solve(*rho, gradient=True, prec="fp32")
    torch.cuda.synchronize()
    g.close()
    for n in range(64):
        g, st = prepared_after(yy, spec, n)
        if st == yy.YY_OK:   # fewer allocations than n
            g.close()
            break
        assert st == yy.YY_ERR_OOM
        with pytest.raises(yy.YYError) as refused:
            g.solve(*rho, gradient=True, prec="fp32")
        assert refused.value.status == yy.YY_ERR_NOT_SUPPORTED
        g.prepare("fp32")
        got = g.solve(*rho, gradient=True, prec="fp32")
        torch.cuda.synchronize()
        assert yy.yy_last_device_status(g.handle) == yy.YY_OK
        for key in ref:
            assert torch.equal(got[key], ref[key]), (n, key)
        g.close()
    assert 6 <= n < 64
