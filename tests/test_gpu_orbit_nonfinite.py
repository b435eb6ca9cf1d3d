"""Samples and pixels that are not finite stay on the rays that meet them
(pytest -m gpu): through the orbit pair as through the general one, they reach
the pixels (rays) that the ray (pixel) has a length in and at most those next
to them, where the walk's second overlap is zero.  (A ray just outside the image
has pixels next to it: the oracle's lengths are those of an image two pixels
wider, on the same rays.)"""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"
GEOMS = [inputs.Geometry(64, 1.1, 16, 64), inputs.Geometry(97, 1.1, 36, 200), inputs.Geometry(70, 1.1, 18, 91),
         inputs.Geometry(70, 1.1, 17, 91)]
IDS = ["8_frames", "8_frames_dense", "4_frames", "general"]


def around(m):
    """A mask with the next pixel along each axis."""
    p = np.pad(m, 1)
    return m | p[:-2, 1:-1] | p[2:, 1:-1] | p[1:-1, :-2] | p[1:-1, 2:]


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")], ids=["nan", "inf", "minf"])
@pytest.mark.parametrize("g", GEOMS, ids=IDS)
def test_backprojection_of_a_sample(g, value):
    wide = dataclasses.replace(g, n=g.n + 2, dgamma=g.fan_pitch)
    og = oracle.Geometry(**{k: getattr(wide, k) for k in oracle.Geometry.__dataclass_fields__})
    plan = air.Plan(g)
    Y = np.random.default_rng(1).random((g.n_views, g.n_bins)).astype(np.float32)
    X, clean = torch.empty(g.n, g.n, device=DEV), torch.empty(g.n, g.n, device=DEV)
    air.air_backproject(plan, torch.as_tensor(Y, device=DEV), clean)
    clean = clean.cpu().numpy()
    for ray in np.random.default_rng(2).permutation(Y.size)[:12]:
        one = np.zeros(Y.size)
        one[ray] = 1.0
        length = oracle.backproject(og, one.reshape(Y.shape)).reshape(g.n + 2, g.n + 2)
        Yv = Y.ravel().copy()
        Yv[ray] = value
        air.air_backproject(plan, torch.as_tensor(Yv, device=DEV), X)
        got = X.cpu().numpy()
        bad = ~np.isfinite(got)
        assert np.all(bad[length[1:-1, 1:-1] > 1e-5])
        assert not np.any(bad & ~around(length > 0)[1:-1, 1:-1])
        assert np.max(np.abs(got - clean)[~bad]) <= 2e-6 * np.max(np.abs(clean))      # one application's tolerance


@pytest.mark.parametrize("value", [float("nan"), float("inf")], ids=["nan", "inf"])
@pytest.mark.parametrize("g", GEOMS, ids=IDS)
def test_projection_of_a_pixel(g, value):
    og = oracle.Geometry(**{k: getattr(g, k) for k in oracle.Geometry.__dataclass_fields__})
    plan = air.Plan(g)
    X = np.random.default_rng(1).random((g.n, g.n)).astype(np.float32)
    A = torch.empty(g.n_views, g.n_bins, device=DEV)
    for k in range(8):
        y, x = np.random.default_rng(k).integers(0, g.n, 2)
        one = np.zeros((g.n, g.n))
        one[y, x] = 1.0
        Xv = X.copy()
        Xv[y, x] = value
        air.air_project(plan, torch.as_tensor(Xv, device=DEV), A)
        bad = ~np.isfinite(A.cpu().numpy())
        here, near = (oracle.project(og, m.astype(np.float64)).reshape(A.shape) for m in (one, around(one > 0)))
        assert np.all(bad[here > 1e-5])
        assert not np.any(bad & ~(near > 0))
