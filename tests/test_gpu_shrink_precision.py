"""The shrink's residual norm to FP64's precision: ||W X - d|| of the FP32
coefficients, against exact arithmetic (pytest -m gpu)."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1310_1434_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air

DEV = "cuda:0"
# the squares are summed without a rounding error above 2^-60, and then take
# at most ten FP64 roundings of 2^-53 each before the root, which halves them
# and adds its own
TOL = 6 * 2.0 ** -53


@pytest.mark.parametrize("n", [1, 2, 3, 31])
def test_residual_norm_is_fp64(n):
    plan = air.Plan(inputs.Geometry(n, 1.0, 8, 16))
    rng = np.random.default_rng(n)
    tau = np.float32(3e-3)
    r, W, g = torch.zeros(1, dtype=torch.float64, device=DEV), torch.empty(9, n, n, device=DEV), torch.empty(n, n, device=DEV)
    for _ in range(40 if n < 4 else 2):
        X = (rng.random((n, n)) * 0.02).astype(np.float32)
        b = ((rng.random((9, n, n)) * 2 - 1) * 0.01).astype(np.float32)
        Xd, bd = torch.as_tensor(X, device=DEV), torch.as_tensor(b, device=DEV)
        air.air_framelet(plan, Xd, W, False)
        air.air_shrink(plan, Xd, bd, g, float(tau), r)
        torch.cuda.synchronize()
        w = W.cpu().numpy()
        t = w + b
        d = np.copysign(np.maximum(np.abs(t) - tau, np.float32(0)), t)
        d[0] = t[0]
        exact = sum((Fraction(float(x)) - Fraction(float(y))) ** 2 for x, y in zip(w.ravel(), d.ravel()))
        assert abs(Fraction(float(r[0])) ** 2 / exact - 1) <= 2 * TOL
