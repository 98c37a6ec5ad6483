"""A walk level of few sinks gives each sink a block of warps, a level of many gives each a warp; both
take the sink's queue in the same order, so its lists and forces must be the same bit for bit.

Two hundred boxes solved together have levels of both kinds, while each box solved alone has few
sinks on every level and is walked by blocks throughout: the forces of the two must agree bit for
bit.  The boxes include sizes around the bucket and group sizes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding, synth

pytestmark = pytest.mark.gpu

TEAM_LEVEL = 4 * 912  # sinks per level from which a GB300's walk gives every sink a warp


def t(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a).reshape(-1)).to("cuda:0", dtype)


def _network():
    """Untrained weights whose predictions straddle the budget: only the two orders are compared."""
    from oracle import mlp as omlp

    rng = np.random.default_rng(4)
    flat = np.zeros(omlp.N_PARAMS)
    flat[:omlp.N_WEIGHTS] = 0.25 * rng.standard_normal(omlp.N_WEIGHTS)
    p = omlp.unpack(flat)
    p["mean"][:] = rng.standard_normal(8)
    p["inv_std"][:] = 0.5 + rng.random(8)
    return omlp.pack(p).astype(np.float32)


@pytest.mark.parametrize("criterion", [0, 1])
def test_many_boxes_equal_each_box_alone(criterion):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sizes = [k for i, small in enumerate((1, 2, 16, 17, 64, 65, 129)) for k in (small, 1500 + i)]
    sizes += [2000 + 23 * i for i in range(186)]
    boxes = [synth.clustered_plummer(k, 300 + i) for i, k in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pos = t(np.concatenate([b[0] for b in boxes], axis=1), torch.float64)
    mass = t(np.concatenate([b[1] for b in boxes]), torch.float32)
    n, eps, theta = int(off[-1]), 1e-3, 0.6
    many, one = binding.Context(0), binding.Context(0)
    try:
        est = torch.zeros(3 * n, dtype=torch.float32, device="cuda:0")
        many.compute_forces_batch(pos, mass, off, eps, theta, est)
        if criterion:
            for c in (many, one):
                c.mlp_load(_network())
                c.set_params(criterion=1, mlp_tau=-3.5)
        acc, pot = est.clone(), torch.zeros(n, dtype=torch.float32, device="cuda:0")
        many.compute_forces_batch(pos, mass, off, eps, theta, acc, pot)
        torch.cuda.synchronize()
        level = many.export_walk_levels()[:, 0]
        assert level.max() >= TEAM_LEVEL > level[level > 0].min()
        if criterion:
            assert many.stats()["n_learned"] > 0
        acc, pot, est = acc.view(3, n), pot, est.view(3, n)
        for b in list(range(16)) + [90, 150, 199]:
            lo, hi = int(off[b]), int(off[b + 1])
            a1 = est[:, lo:hi].contiguous().view(-1)
            p1 = torch.zeros(hi - lo, dtype=torch.float32, device="cuda:0")
            one.compute_forces(t(boxes[b][0], torch.float64), t(boxes[b][1], torch.float32), eps, theta, a1, p1)
            torch.cuda.synchronize()
            assert torch.equal(acc[:, lo:hi], a1.view(3, -1)) and torch.equal(pot[lo:hi], p1), b
    finally:
        many.close()
        one.close()
