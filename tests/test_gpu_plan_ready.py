"""A plan is ready when air_plan_create returns: its first call may come at once,
on a stream that waits for nothing else, while other work fills the GPU
(pytest -m gpu).  The first plan of a geometry is tuned, which waits for the
device; the plans after it are not, so they show whether creation itself does."""
import dataclasses

import pytest

from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"
# with orbits, and without
GEOMS = [inputs.Geometry(256, 1.6, 200, 384), inputs.Geometry(256, 1.6, 201, 384)]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("g", GEOMS, ids=["orbits", "general"])
@pytest.mark.parametrize("op", ["project", "backproject", "fbackproject", "solve"])
def test_first_call_right_after_creation(g, prec, op):
    g = dataclasses.replace(g, precision=prec)
    gen = torch.Generator(DEV).manual_seed(3)
    X = torch.rand(g.n, g.n, device=DEV, generator=gen)
    Y = torch.rand(g.n_views, g.n_bins, device=DEV, generator=gen)

    def call(plan, out, stream):
        if op == "project":
            air.air_project(plan, X, out, stream)
        elif op == "backproject":
            air.air_backproject(plan, Y, out, stream)
        elif op == "fbackproject":
            air.air_filtered_backproject(plan, Y, out, stream)
        else:
            air.air_solve(plan, Y, 1e-3, 1.0, 1, 2, out, None, stream)

    side, busy = torch.cuda.Stream(), torch.cuda.Stream()
    ref, *outs = [torch.full_like(Y if op == "project" else X, float("nan")) for _ in range(5)]
    torch.cuda.synchronize()
    first = air.Plan(g)
    call(first, ref, side)
    load = air.Plan(inputs.Geometry(512, 0.8, 801, 738))     # its projections fill the GPU
    big, sino = torch.rand(512, 512, device=DEV), torch.empty(801, 738, device=DEV)
    torch.cuda.synchronize()
    for out in outs:
        for _ in range(10):
            air.air_project(load, big, sino, busy)
        plan = air.Plan(g)
        call(plan, out, side)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
