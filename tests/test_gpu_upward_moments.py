"""Moments, masses, boxes and active counts of the tree's cells against sums over their particles, for trees in
which a warp of the upward pass goes on with many lanes, with few (it then computes their cells
together) and down long one-sided chains.

The GPU adds a bucket's moments in FP32 and shifts them level by level, about a dozen roundings of 6e-8
each per level, relative to M b_max^n at most: 3e-5 of that for the 40 levels of the deepest tree here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def _chain(n, seed):
    rng = np.random.default_rng(seed)
    return rng.random((3, n)) * 0.999 * 2.0 ** -rng.integers(0, 12, n), np.full(n, 1.0 / n, np.float32)


@pytest.mark.parametrize("n,kind,bucket", [(17, "plummer", 16), (33, "plummer", 16), (40, "chain", 1), (700, "plummer", 16),
                                           (3000, "chain", 16), (20000, "plummer", 8)])
def test_cells_match_sums_over_their_particles(n, kind, bucket):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pos, mass = _chain(n, 5) if kind == "chain" else synth.clustered_plummer(n, 21)
    active = (np.arange(n) % 3 != 0).astype(np.uint8)
    ctx = binding.Context(0, bucket=bucket)
    try:
        ctx.build_tree(torch.from_numpy(pos.reshape(-1).copy()).cuda(), torch.from_numpy(mass).cuda(),
                       torch.from_numpy(active).cuda())
        perm, _ = ctx.export_order(n)
        c = ctx.export_cells()
    finally:
        ctx.close()
    # slots of a moment record: 1, then the monomials of orders 2 to 4, first axis' power falling
    mono = [(0, 0, 0)] + [(o - m, m - k, k) for o in (2, 3, 4) for m in range(o + 1) for k in range(m + 1)]
    x, m64, act = pos[:, perm], mass[perm].astype(np.float64), active[perm]
    assert (c["child"][:, 0] >= 0).any()
    for i in range(len(c["first"])):
        s = slice(int(c["first"][i]), int(c["first"][i]) + int(c["count"][i]))
        M = m64[s].sum()
        com = (x[:, s] * m64[s]).sum(1) / M
        assert abs(c["mass"][i] - M) <= 1e-13 * M and np.abs(c["com"][i] - com).max() <= 1e-12
        assert np.array_equal(c["lo"][i], x[:, s].min(1)) and np.array_equal(c["hi"][i], x[:, s].max(1))
        assert c["nact"][i] == act[s].sum()
        y = x[:, s] - c["com"][i][:, None]
        for slot, (a, b, k) in enumerate(mono):
            want = (m64[s] * y[0] ** a * y[1] ** b * y[2] ** k).sum()
            scale = M * max(float(c["bmax"][i]), 1e-300) ** (a + b + k)
            assert abs(c["moments"][i, slot] - want) <= 3e-5 * scale + 1e-37, (i, slot)
