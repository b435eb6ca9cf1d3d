"""Batch tables are copied on the stream that runs the batch: a new batch on a
stream that waits for no other gives the same images in both forms, with work
on the default stream beside it (pytest -m gpu)."""
import pytest

from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"


@pytest.mark.parametrize("form", ["grouped", "persistent"])
def test_new_batch_on_a_side_stream(form):
    gs = [inputs.Geometry(64, 1.2, 32, 96), inputs.Geometry(48, 1.7, 33, 70)]
    f = air.air_solve_batch if form == "grouped" else air.air_solve_batch_persistent
    gen = torch.Generator(DEV).manual_seed(5)
    Ys = [torch.rand(g.n_views * g.n_bins, device=DEV, generator=gen) for g in gs]
    sets = [[torch.full((g.n ** 2,), float("nan"), device=DEV) for g in gs] for _ in range(4)]
    other, side = torch.rand(4096, 4096, device=DEV), torch.cuda.Stream()
    torch.cuda.synchronize()
    for i, Xs in enumerate(sets):               # new plans: a graph of its own each time
        plans = [air.Plan(g) for g in gs]
        for _ in range(i * 5):
            other = other @ other * 1e-3
        f(plans, Ys, [1e-3] * 2, [1.0] * 2, [2, 3], [3, 2], Xs, side)
    torch.cuda.synchronize()
    for Xs in sets:
        assert all(torch.isfinite(x).all() and torch.equal(x, y) for x, y in zip(Xs, sets[0]))
