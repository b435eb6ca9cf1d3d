"""The orbit backprojector's FP32 sums against FP64 (pytest -m gpu)."""
import numpy as np
import pytest

import oracle
from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"
# An FP32 rounding of a value anywhere in its binade is 2.5e-8 of it in the rms
# (2^-24 * 0.42).  A pixel of positive samples takes one at its full size with the
# scale, at most 0.75 more in the mean square for the sums within its images'
# fours, and the partial sums that make an image, an eighth of their views each,
# take less than two more (less the more splits there are).  Together
# sqrt(1 + 0.75 + 2) * 2.5e-8 = 4.8e-8 at the most, and the lengths of nearly
# axis-parallel rays add their 2^-32 px.  Before its first run the bound was
# set at 7e-8, for images added up in a row.
TOL = 7e-8


@pytest.mark.parametrize("g", [inputs.Geometry(128, 1.0, 400, 192), inputs.Geometry(96, 1.3, 300, 150, beta0=0.2),
                               inputs.Geometry(97, 1.3, 400, 150)], ids=["8_frames", "4_frames", "odd"])
def test_backprojection_sums(g):
    og = oracle.Geometry(**{k: getattr(g, k) for k in oracle.Geometry.__dataclass_fields__})
    Y = np.random.default_rng(7).random((g.n_views, g.n_bins)).astype(np.float32)
    ref = oracle.backproject(og, Y.astype(np.float64)).ravel()
    plan = air.Plan(g)
    X = torch.empty(g.n * g.n, device=DEV)
    vpb, _, most = air.air_plan_config(plan)
    for parts in sorted({8, 16, 32, most}):
        air.air_plan_tune(plan, vpb, min(parts, most))
        air.air_backproject(plan, torch.as_tensor(Y, device=DEV), X)
        torch.cuda.synchronize()
        err = np.linalg.norm(X.cpu().numpy().astype(np.float64) - ref) / np.linalg.norm(ref)
        assert err <= TOL, (parts, err)
