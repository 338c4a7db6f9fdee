"""Kernels that start while their predecessors end: the same bits as one after the other.

Profiling runs a solve's kernels strictly in turn, so its results are the reference.  Against
them: solves back to back on a caller's own stream, forms and grids in changing order, each
input written by a kernel just before its solve and each output copied and overwritten by kernels just after."""

import numpy as np
import pytest

from paper_1806_04593_gb300 import inputs
from tests.gpu_common import lib, require_gpu

pytestmark = pytest.mark.gpu

FORMS = [("fp64", "auto"), ("fp64", "dense"), ("fp32", "auto"), ("fp32", "dense"), ("fp64_ozaki", "auto"), ("fp64_ozaki", "dense"),
         ("fp16x2", "auto"), ("fp16x2", "separable"), ("bf16x3", "auto"), ("bf16x3", "separable"), ("tf32", "auto"), ("tf32", "separable")]


def specs():
    r = lambda n: np.logspace(-2, 0, n + 1)  # noqa: E731
    return [inputs.tiny_grid(), inputs.GridSpec("even", r(60), 24, 72, 0.0, 0.0, 12), inputs.GridSpec("odd", r(37), 35, 105, 0.0, 0.0, 33),
            inputs.polar_grid(r(50), 30, 60, 20), inputs.GridSpec("long", r(40), 90, 270, 0.0, 0.0, 10)]


@pytest.mark.parametrize("gradient", [False, True])
def test_back_to_back(gradient):
    require_gpu()
    import torch
    yy = lib()
    runs = []
    for n, spec in enumerate(specs()):
        g = yy.Grid.from_spec(spec)
        for prec in dict.fromkeys(p for p, _ in FORMS):
            g.prepare(prec)
        shape = (spec.n_r, spec.n_theta, spec.n_phi)
        patches = 1 if spec.polar else 2
        gen = torch.Generator(device="cuda").manual_seed(n)
        rho = [1.0 + torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda") for _ in range(patches)]
        io = lambda: [torch.empty(shape, dtype=torch.float64, device="cuda") for _ in range(patches)]  # noqa: E731
        runs.append({"g": g, "rho": rho, "in": io(), "phi": io(), "patches": patches,
                     "grad": [torch.empty((3,) + shape, dtype=torch.float64, device="cuda") for _ in range(patches)] if gradient else None})

    def solve(run, form, stream):
        other = lambda a: a[1] if a is not None and run["patches"] == 2 else None  # noqa: E731
        first = lambda a: None if a is None else a[0]  # noqa: E731
        run["g"].set_analysis(form[1])
        run["g"].potential(run["in"][0], other(run["in"]), run["phi"][0], other(run["phi"]), first(run["grad"]), other(run["grad"]),
                           prec=form[0], stream=stream)

    def outputs(run):
        return run["phi"] + (run["grad"] or [])

    steps = [(k, f) for f in range(len(FORMS)) for k in range(len(runs))]
    ref = {}
    for k, f in steps:
        run = runs[k]
        for a, b in zip(run["in"], run["rho"]):
            torch.mul(b, 1.0 + f, out=a)
        yy.yy_grid_set_profiling(run["g"].handle, 1)
        torch.cuda.synchronize()
        solve(run, FORMS[f], None)
        torch.cuda.synchronize()
        yy.yy_grid_set_profiling(run["g"].handle, 0)
        ref[k, f] = [x.clone() for x in outputs(run)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    got = []
    rng = np.random.default_rng(0)
    with torch.cuda.stream(stream):
        for at in list(rng.permutation(len(steps))) + list(range(len(steps))):
            k, f = steps[at]
            run = runs[k]
            for a, b in zip(run["in"], run["rho"]):
                torch.mul(b, 1.0 + f, out=a)
            solve(run, FORMS[f], stream)
            got.append((k, f, [x.clone() for x in outputs(run)]))
            for x in outputs(run) + run["in"]:
                x.fill_(float("nan"))
    torch.cuda.synchronize()
    for k, f, out in got:
        for x, y in zip(out, ref[k, f]):
            assert torch.equal(x, y), (specs()[k].name, FORMS[f], int((x != y).sum()))
    for run in runs:
        assert yy.yy_last_device_status(run["g"].handle) == yy.YY_OK
        run["g"].close()
