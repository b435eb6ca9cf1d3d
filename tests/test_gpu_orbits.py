"""The projector pair over orbits of rays (full scans with at least four
symmetries) on the GPU: parity with the FP64 oracle at the single-application
tolerance, and A and A^T exact transposes of one another, at ragged tiles, odd
sides and bin counts, both group orders and views a mirror takes to themselves
(pytest -m gpu)."""
import math

import numpy as np
import pytest

import oracle
from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"
TOL_OP = 2e-6     # a single A or A^T application against the oracle

GEOMS = [inputs.Geometry(64, 1.1, 16, 64), inputs.Geometry(77, 1.3, 32, 101), inputs.Geometry(97, 1.1, 36, 64),
         inputs.Geometry(65, 1.1, 18, 91), inputs.Geometry(70, 1.1, 20, 101, beta0=0.2),
         inputs.Geometry(66, 1.0, 20, 95, beta0=math.pi / 20), inputs.Geometry(130, 3.0, 44, 170),
         inputs.Geometry(200, 1.7, 90, 290)]
IDS = [f"{g.n}_{g.n_views}_{g.n_bins}" for g in GEOMS]


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy().astype(np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("g", GEOMS, ids=IDS)
def test_orbit_pair_matches_oracle(g):
    og = oracle.Geometry(**{k: getattr(g, k) for k in oracle.Geometry.__dataclass_fields__})
    X = inputs.random_image(g.n, 5).astype(np.float32)
    Y = inputs.random_sinogram(g.n_views, g.n_bins, 6).astype(np.float32)
    plan = air.Plan(g)
    Xd, Yd = torch.as_tensor(X, device=DEV), torch.as_tensor(Y, device=DEV)
    A, B = torch.full_like(Yd, float("nan")), torch.full_like(Xd, float("nan"))
    A_ref, B_ref = oracle.project(og, X.astype(np.float64)), oracle.backproject(og, Y.astype(np.float64))
    vpb, _, most = air.air_plan_config(plan)
    for parts in sorted({1, 8, max(8, most // 2), most}):
        air.air_plan_tune(plan, vpb, parts)
        air.air_project(plan, Xd, A)
        air.air_backproject(plan, Yd, B)
        torch.cuda.synchronize()
        assert rel(A, A_ref.reshape(A.shape)) <= TOL_OP and rel(B, B_ref.reshape(B.shape)) <= TOL_OP, parts


@pytest.mark.parametrize("g", [GEOMS[0], GEOMS[3]], ids=[IDS[0], IDS[3]])
def test_orbit_pair_is_exactly_adjoint(g):
    # sampled rows and columns of A hold the same FP32 lengths, bit for bit
    plan = air.Plan(g)
    nn, m = g.n * g.n, g.n_views * g.n_bins
    rng = np.random.default_rng(0)
    px, ray = rng.permutation(nn)[:300], rng.permutation(m)[:300]
    A, AT = torch.empty(m, device=DEV), torch.empty(nn, device=DEV)
    a, at = np.zeros((300, 300), np.float32), np.zeros((300, 300), np.float32)
    for i, p in enumerate(px):
        e = torch.zeros(nn, device=DEV)
        e[int(p)] = 1.0
        air.air_project(plan, e, A)
        a[:, i] = A.cpu().numpy()[ray]
    for i, q in enumerate(ray):
        e = torch.zeros(m, device=DEV)
        e[int(q)] = 1.0
        air.air_backproject(plan, e, AT)
        at[i] = AT.cpu().numpy()[px]
    assert np.array_equal(a, at)
    assert (a != 0).sum() > 300


@pytest.mark.parametrize("prec", [0, 1])
def test_orbit_solve_matches_oracle(prec):
    # without a residual history the solve runs the orbit pair
    w = inputs._wl("orbit_solve", 100, 1.1, 40, 150, 11, 6, 3, 1e5, n_outer=3, n_cg=4, precision=prec)
    Y = inputs.make_case(w)[2].astype(np.float32)
    og = oracle.Geometry(**{k: getattr(w.geom, k) for k in oracle.Geometry.__dataclass_fields__})
    ref = oracle.solve(og, Y.astype(np.float64), w.lam, w.mu, w.n_outer, w.n_cg)
    plan = air.Plan(w.geom)
    X = torch.empty(w.geom.n, w.geom.n, device=DEV)
    air.air_solve(plan, torch.as_tensor(Y, device=DEV), w.lam, w.mu, w.n_outer, w.n_cg, X)
    torch.cuda.synchronize()
    assert rel(X, ref.reshape(X.shape)) <= 1e-4


FBP_GEOMS = GEOMS + [inputs.Geometry(33, 2.0, 30, 41), inputs.Geometry(40, 2.0, 26, 50, beta0=math.pi / 26),
                     inputs.Geometry(17, 3.0, 4, 31), inputs.Geometry(50, 1.1, 24, 64, dso_mm=60.0)]


@pytest.mark.parametrize("g", FBP_GEOMS, ids=[f"{g.n}_{g.n_views}_{g.n_bins}" for g in FBP_GEOMS])
def test_orbit_fbp_matches_oracle(g):
    # the analytic reconstruction over orbits of views, at the tolerance
    # derived for the general one (FP32 sum over the views and 2e-5 bins of
    # interpolation position): 5e-6
    og = oracle.Geometry(**{k: getattr(g, k) for k in oracle.Geometry.__dataclass_fields__})
    Y = inputs.ellipse_line_integrals(g, inputs.random_phantom(g, 3, 6, 3)).astype(np.float32)
    plan = air.Plan(g)
    X = torch.full((g.n, g.n), float("nan"), device=DEV)
    air.air_fbp(plan, torch.as_tensor(Y, device=DEV), X)
    torch.cuda.synchronize()
    assert rel(X, oracle.fbp(og, Y.astype(np.float64)).reshape(X.shape)) <= 5e-6
