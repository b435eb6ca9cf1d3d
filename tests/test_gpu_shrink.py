"""The fused shrink at the edges of its 30 x 6 tiles and of its two-float sum of
squares (pytest -m gpu): against the FP64 oracle, and scaled by powers of two,
which FP32 carries through exactly, beyond the range of FP32 squares."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1310_1434_gb300 import air, inputs

DEV = "cuda:0"


def shrink(n, X, b, tau):
    plan = air.Plan(inputs.Geometry(n, 1.0, 8, 16))
    bd, g = torch.as_tensor(b, device=DEV), torch.full((n, n), float("nan"), device=DEV)
    r = torch.zeros(1, dtype=torch.float64, device=DEV)
    air.air_shrink(plan, torch.as_tensor(X, device=DEV), bd, g, tau, r)
    torch.cuda.synchronize()
    return bd.cpu().numpy(), g.cpu().numpy(), float(r[0])


@pytest.mark.parametrize("n", [1, 2, 30, 31, 60, 97, 769])
def test_shrink_tiles_and_range(n):
    rng = np.random.default_rng(n)
    X = (rng.random((n, n)) * 0.02).astype(np.float32)
    tau = float(np.float32(3e-4))
    b = ((rng.random((9, n, n)) * 2 - 1) * tau).astype(np.float32)
    got_b, got_g, got_r = shrink(n, X, b, tau)
    ref_b, ref_g, ref_r = oracle.shrink(X.astype(np.float64), b.astype(np.float64), tau)
    # values of 0.02 at most through a few FP32 roundings of 2^-24 each; a
    # coefficient at the threshold may fall on either side, which is continuous
    assert np.max(np.abs(got_b - np.asarray(ref_b).reshape(b.shape))) <= 2e-8
    assert np.max(np.abs(got_g - np.asarray(ref_g).reshape(X.shape))) <= 2e-7
    assert abs(got_r - ref_r) <= 1e-6 * ref_r + 1e-12
    for e in (-90, 80):                        # squares of 2^-180 and 2^160 leave FP32
        s = np.float32(2.0) ** np.float32(e)
        sb, sg, sr = shrink(n, X * s, b * s, float(np.float32(tau) * s))
        assert np.array_equal(sb, got_b * s) and np.array_equal(sg, got_g * s)
        assert abs(sr - got_r * float(s)) <= 1e-12 * got_r * float(s)
