"""Tensor-core filter at the edges of its split kernel and of its K loop, and a
solve that stops at once (pytest -m gpu).

Bound of a single application: 2e-6 relative L2 against the FP64 oracle, the
one the other filter tests hold it to (24-bit splits and FP32 sums of a few
hundred terms grouped by magnitude stay below 5e-7; the rest is margin)."""
import numpy as np
import pytest

import oracle
from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"


# bins: fewer than a thread's eight, around the near band's 64 lags and the
# padding to 128, odd (rows off 8-byte boundaries); one to five chunks of K
# (fewer than, as many as and more than the stage ring); views around a tile
@pytest.mark.parametrize("views,bins", [(1, 5), (3, 63), (5, 65), (127, 128), (129, 129), (7, 383), (128, 385),
                                        (130, 513), (2, 639)])
def test_filter_edges(views, bins):
    g = inputs.Geometry(8, 1.0, views, bins, precision=1)
    Y = np.random.default_rng(bins).random((views, bins), dtype=np.float32)
    plan = air.Plan(g)
    Yd = torch.as_tensor(Y.ravel(), device=DEV)
    Zd = torch.full((views * bins + 1,), 7.0, device=DEV)
    air.air_filter(plan, Yd, Zd[:-1])
    air.air_plan_status(plan)
    og = oracle.Geometry(**{k: getattr(g, k) for k in oracle.Geometry.__dataclass_fields__})
    ref = oracle.filter(og, Y.astype(np.float64)).ravel()
    out = Zd.cpu().numpy()
    assert out[-1] == 7.0
    assert np.linalg.norm(out[:-1] - ref) <= 2e-6 * np.linalg.norm(ref)


def test_stopped_solve_leaves_the_filter_usable():
    """From zeros CG stops before its first filter, whose products are then
    skipped with their first operands already on the way."""
    g = inputs.Geometry(32, 2.0, 13, 400, precision=1)
    plan = air.Plan(g)
    Y = torch.rand(13 * 400, device=DEV)
    before, after, X = torch.empty_like(Y), torch.empty_like(Y), torch.full((32 * 32,), 7.0, device=DEV)
    air.air_filter(plan, Y, before)
    air.air_solve(plan, torch.zeros_like(Y), 1e-3, 1e-2, 2, 3, X)
    air.air_filter(plan, Y, after)
    air.air_plan_status(plan)
    assert torch.count_nonzero(X) == 0
    assert torch.equal(before, after)
