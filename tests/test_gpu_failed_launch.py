"""A solve whose launches the runtime refuses returns an error and leaves none behind.

The refusal is the host's: the stream's capture has been invalidated (by an
allocation, which a global capture forbids), so no launch into it is accepted and nothing
runs.  The calls after it, on other grids, do as they always do."""

import ctypes

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp64_ozaki", "fp16x2"])
def test_refused_launches(prec):
    require_gpu()
    import torch
    yy = lib()
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    spec = inputs.tiny_grid()
    rho = [torch.as_tensor(x, device="cuda") for x in inputs.density_for(spec)]
    out = [torch.empty_like(x) for x in rho]
    g = yy.Grid.from_spec(spec)
    g.prepare(prec)
    g.potential(rho[0], rho[1], out[0], out[1], prec=prec)
    torch.cuda.synchronize()
    before = [x.cpu().numpy() for x in out]
    stream, graph, mem = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamCreateWithFlags(ctypes.byref(stream), 1) == 0
    assert rt.cudaStreamBeginCapture(stream, 0) == 0
    assert rt.cudaMalloc(ctypes.byref(mem), ctypes.c_size_t(16)) != 0
    try:
        with pytest.raises(yy.YYError):
            g.potential(rho[0], rho[1], out[0], out[1], prec=prec, stream=stream.value)
    finally:
        assert rt.cudaStreamEndCapture(stream, ctypes.byref(graph)) != 0
        rt.cudaGetLastError()
        assert rt.cudaStreamDestroy(stream) == 0
    other = yy.Grid.from_spec(spec)
    other.prepare(prec)
    other.potential(rho[0], rho[1], out[0], out[1], prec=prec)
    torch.cuda.synchronize()
    for x, y in zip(out, before):
        assert np.array_equal(x.cpu().numpy(), y)
    g.potential(rho[0], rho[1], out[0], out[1], prec=prec)
    torch.cuda.synchronize()
    for x, y in zip(out, before):
        assert np.array_equal(x.cpu().numpy(), y)
    for h in (g, other):
        assert yy.yy_last_device_status(h.handle) == yy.YY_OK
        h.close()
