"""Orbits cost a plan memory: a server budget that holds the plan without them
still serves the request (pytest -m gpu)."""
import numpy as np
import pytest

from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air


@pytest.mark.parametrize("g,twin", [
    # every symmetry, but a ray along a grid line: no orbit tables
    (inputs.Geometry(66, 1.0, 40, 101), inputs.Geometry(66, 1.0, 40, 101)),
    # orbit tables, against the same sizes without a symmetry
    (inputs.Geometry(130, 2.0, 42, 170), inputs.Geometry(130, 2.0, 42, 170, beta0=0.01)),
    (inputs.Geometry(130, 2.0, 42, 170, precision=1), inputs.Geometry(130, 2.0, 42, 170, beta0=0.01, precision=1)),
], ids=["declined", "orbits", "orbits_bf16x3"])
def test_budget_of_the_general_path_is_enough(g, twin):
    Y = inputs.noisy_sinogram(inputs.ellipse_line_integrals(g, inputs.random_phantom(g, 12, 6, 2)), 2e4, 12)
    Y = Y.astype(np.float32).ravel()
    X = torch.empty(g.n * g.n, device="cuda")
    air.air_solve(air.Plan(g), torch.as_tensor(Y, device="cuda"), 3e-4, 1.0, 4, 2, X)
    ref = X.cpu().numpy()
    srv = air.Server(int(air.Plan(twin).nbytes * 1.01), max_slots=4)
    ids = [srv.submit(g, Y, 3e-4, 1.0, 4, 2) for _ in range(2)]
    for rid in ids:
        X = srv.wait(rid, g.n)
        assert np.linalg.norm(X - ref) <= 1e-4 * np.linalg.norm(ref)
    srv.close()
