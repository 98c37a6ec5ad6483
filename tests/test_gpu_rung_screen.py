"""The kick-drift's rungs are decided in FP32 away from the thresholds and in FP64 near them: both must
give the oracle's FP64 rungs exactly, for accelerations at the thresholds to the last bit, over all
magnitudes FP32 holds, and for time steps whose thresholds leave FP32's range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import kdk
from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps,dt0,R", [(1e-3, 1e-2, 5), (7.8e-5, 3e-3, 1), (1e-3, 0.3, 30), (1e-12, 1e-14, 8),
                                       (1e-3, 1e-30, 4), (1e-3, 1e12, 30)])
def test_rungs_at_the_thresholds(eps, dt0, R):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(R)
    n = 200_003
    # |a| whose Delta T is dt0 2^-k, and its neighbourhood from one part in 10^9 to one in 10^3
    k = rng.integers(-1, R + 2, n)
    with np.errstate(over="ignore"):
        am = 0.04 * eps / (dt0 * 2.0 ** -k.astype(float)) ** 2
    am *= 1.0 + rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-9, -3, n) * (rng.random(n) < 0.9)
    wide = rng.random(n) < 0.3
    am[wide] = 10.0 ** rng.uniform(-44, 38, int(wide.sum()))
    d = rng.standard_normal((3, n))
    d[:, ::7] = [[1.0], [0.0], [0.0]]
    with np.errstate(over="ignore", under="ignore"):
        acc = (d / np.linalg.norm(d, axis=0) * am).astype(np.float32)
    acc[:, :3] = 0.0
    acc[0, 3] = np.inf
    acc[:, 4] = 1e-45
    with np.errstate(all="ignore"):
        want = kdk.target_rungs(acc, eps, dt0, R)
    ctx = binding.Context(0)
    try:
        rung = torch.zeros(n, dtype=torch.uint8, device="cuda:0")
        ctx.assign_rungs(torch.from_numpy(acc.reshape(-1)).cuda(), rung, eps, dt0, R)
        torch.cuda.synchronize()
        assert np.array_equal(rung.cpu().numpy(), want)
    finally:
        ctx.close()
