"""Kick-drift with a single rung: every particle is active and is kicked in its own lane, where several rungs gather
the active ones.  Against the oracle's schedule (FP64 updates that may differ by the rounding of one fused
multiply-add, relative 1e-15), and against the gathering kernel's velocities bit for bit (two rungs, all
particles on the coarse one and slow enough to stay there).  Particles that come from finer rungs are closed
with their own half step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import kdk
from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("closing", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 255, 256, 257, 50_000])
def test_single_rung(n, closing):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    pos = 0.25 + 0.5 * rng.random((3, n))
    vel = 1e-3 * rng.standard_normal((3, n))
    acc = rng.uniform(-1.0, 1.0, (3, n)).astype(np.float32)
    acc[:, 0] = 0.0
    eps, dt0 = 1e-3, 1e-3  # 0.2 sqrt(eps / |a|) > 4 dt0: rung 0 whatever the number of rungs
    ctx = binding.Context(0)

    def step(R, rungs=None):
        t = [torch.from_numpy(a.reshape(-1).copy()).cuda() for a in (pos, vel, acc)]
        rung, nxt = (torch.zeros(n, dtype=torch.uint8, device="cuda:0") for _ in range(2))
        nxt.fill_(9)
        if rungs is not None:
            rung.copy_(torch.from_numpy(rungs.astype(np.uint8)))
        ctx.kick_drift(t[0], t[1], t[2], rung, nxt, eps, dt0, R, 0, closing)
        torch.cuda.synchronize()
        return t[0].cpu().numpy().reshape(3, n), t[1].cpu().numpy().reshape(3, n), rung.cpu().numpy(), nxt.cpu().numpy()

    try:
        p, v, r, a = step(0)
        p2, v2, r2, a2 = kdk.kick_drift(pos, vel, acc, np.zeros(n, np.int64), eps, dt0, 0, 0, closing)
        assert np.array_equal(r, r2) and np.array_equal(a.astype(bool), a2) and (a == 1).all()
        assert np.allclose(v, v2, rtol=1e-15, atol=1e-18) and np.allclose(p, p2, rtol=1e-15, atol=1e-18)
        # a step that ends finer rungs: their closing half step, then the single rung
        fine = rng.integers(0, 5, n)
        p, v, r, a = step(0, fine)
        w = vel.copy()
        if closing:
            w += acc.astype(np.float64) * (dt0 * 2.0 ** -(fine + 1.0))
        w += acc.astype(np.float64) * (0.5 * dt0)
        assert not r.any() and (a == 1).all() and np.allclose(v, w, rtol=1e-15, atol=1e-18)
        p, v, r, a = step(0)
        _, w, r1, _ = step(1)
        assert not r1.any() and np.array_equal(v, w)
    finally:
        ctx.close()
