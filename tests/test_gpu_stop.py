"""Solves whose CG stops at once: every phase then reads its operands together
with the stop flag and must leave all of them alone (pytest -m gpu).  A zero
sinogram gives a zero image exactly, and a solve after it gives the bits of the
one before."""
import pytest

from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"

# a full symmetry group, half of it, and a scan without (the general path);
# 70 is not a multiple of a tile, and 128 has launches of a few blocks
GEOMS = [inputs.Geometry(128, 1.0, 96, 192), inputs.Geometry(70, 2.0, 90, 120), inputs.Geometry(70, 2.0, 45, 120)]


@pytest.mark.parametrize("g", GEOMS, ids=lambda g: f"{g.n}_v{g.n_views}")
@pytest.mark.parametrize("form", ["solve", "history", "l2", "batch", "persistent"])
def test_stopped_solve(g, form):
    plan = air.Plan(g)
    hist = torch.zeros(2, dtype=torch.float64, device=DEV)

    def run(Y):
        X = torch.full((g.n * g.n,), 7.0, device=DEV)
        if form == "solve":
            air.air_solve(plan, Y, 1e-3, 1e-2, 2, 3, X)
        elif form == "history":
            air.air_solve(plan, Y, 1e-3, 1e-2, 2, 3, X, hist)
        elif form == "l2":
            air.air_solve_l2(plan, Y, 1e-2, 3, X)
        else:
            f = air.air_solve_batch if form == "batch" else air.air_solve_batch_persistent
            f([plan], [Y], [1e-3], [1e-2], [2], [3], [X])
        air.air_plan_status(plan)
        return X

    Y = torch.rand(g.n_views * g.n_bins, device=DEV, generator=torch.Generator(DEV).manual_seed(1))
    before = run(Y)
    assert torch.count_nonzero(before) > 0
    assert torch.count_nonzero(run(torch.zeros_like(Y))) == 0
    assert torch.equal(run(Y), before)
