"""Batch graphs serve calls with other sinograms, images and weights, other
plans of the same shapes, and more compositions than are kept (pytest -m gpu)."""
import numpy as np
import pytest

from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"


def workloads(prec):
    return [inputs._wl("r0", 64, 1.2, 32, 96, 3, 5, 2, 1e5, n_outer=2, n_cg=3, precision=prec),
            inputs._wl("r1", 48, 1.7, 33, 70, 4, 5, 2, 1e5, n_outer=3, n_cg=2)]


def check(ws, plans, seed, lam, stream=None):
    Ys = [torch.as_tensor(inputs.make_case(w)[2].astype(np.float32).ravel() * (1.0 + 0.1 * seed), device=DEV) for w in ws]
    Xs = [torch.full((w.geom.n ** 2,), float("nan"), device=DEV) for w in ws]
    torch.cuda.synchronize()
    air.air_solve_batch(plans, Ys, [lam] * 2, [1.0] * 2, [w.n_outer for w in ws], [w.n_cg for w in ws], Xs, stream)
    for w, p, y, x in zip(ws, plans, Ys, Xs):
        ref = torch.empty_like(x)
        air.air_solve(p, y, lam, 1.0, w.n_outer, w.n_cg, ref)
        torch.cuda.synchronize()
        # the same kernels in the same order
        assert torch.equal(x, ref), (w.name, seed, lam)


@pytest.mark.parametrize("prec", [0, 1])
def test_graphs_serve_other_data_plans_and_streams(prec):
    ws = workloads(prec)
    sets = [[air.Plan(w.geom) for w in ws] for _ in range(2)]
    side = torch.cuda.Stream()
    for seed in range(4):                       # two compositions in turn, new buffers each time
        check(ws, sets[seed % 2], seed, 1e-3 * (seed + 1), side if seed > 1 else None)
    graph = air.air_batch_graph_info()
    for p in sets.pop(0):                       # a plan's graphs go with it
        p.close()
    check(ws, sets[0], 7, 2e-3)
    assert air.air_batch_graph_info() == graph
    more = [[air.Plan(w.geom) for w in ws] for _ in range(9)]      # one more than are kept
    for i, plans in enumerate(more + more[:1]):
        check(ws, plans, i, 1e-3)


def test_plans_that_take_a_destroyed_plans_place():
    # a new plan may get the address of a destroyed one, and its buffers those
    # of freed ones: the destroyed plan's graph must not serve it
    ws = workloads(1)
    for seed in range(4):
        plans = [air.Plan(w.geom) for w in ws]
        check(ws, plans, seed, 1e-3)
        pad = torch.empty((seed + 1) << 22, device=DEV)     # shifts what the next plans are given
        for p in plans:
            p.close()
        del pad
