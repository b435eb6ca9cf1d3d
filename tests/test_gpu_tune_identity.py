"""Setting a plan's configuration as it was read changes nothing, and on a scan
with orbits the images of their backprojector are not the view parts of the
general pair, which its solves with a residual history run (pytest -m gpu)."""
import pytest

from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"


@pytest.mark.parametrize("g", [inputs.Geometry(128, 1.0, 90, 192), inputs.Geometry(128, 1.0, 91, 192)],
                         ids=["orbits", "general"])
def test_config_then_tune_is_the_identity(g):
    plan = air.Plan(g)
    Y = torch.rand(g.n_views * g.n_bins, device=DEV, generator=torch.Generator(DEV).manual_seed(1))

    def history():
        X, r = torch.empty(g.n * g.n, device=DEV), torch.zeros(2, dtype=torch.float64, device=DEV)
        air.air_solve(plan, Y, 1e-3, 1.0, 2, 3, X, r)
        return X, r

    vpb, parts, most = air.air_plan_config(plan)
    ref = history()
    air.air_plan_tune(plan, vpb, parts)
    assert air.air_plan_config(plan) == (vpb, parts, most)
    assert all(torch.equal(a, b) for a, b in zip(history(), ref))
    if g.n_views % 2 == 0:                      # (with orbits)
        for s in (1, 8, most):                  # images of the orbit pair alone
            air.air_plan_tune(plan, vpb, s)
            assert air.air_plan_config(plan)[1] == max(8, s // 8 * 8)
            assert all(torch.equal(a, b) for a, b in zip(history(), ref))
