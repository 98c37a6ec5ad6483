"""A walk of a million cells or more keeps each level's sinks in tree order; a smaller one takes them
as they come.  Neither changes a sink's lists or the order within them, so the forces must be the same
bit for bit: many boxes solved together (in order) against each box alone (as they come), with every
particle active and with a part of them (cells with one active child, or none)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding, synth

pytestmark = pytest.mark.gpu

ORDERED = 1 << 20  # cells from which a walk keeps its sinks in order


@pytest.mark.parametrize("every", [1, 3])
def test_ordered_sinks_give_the_same_forces(every):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    base = [synth.clustered_plummer(7000 + 37 * i, 500 + i) for i in range(24)]
    boxes = [base[i % 24] for i in range(240)]
    off = np.concatenate([[0], np.cumsum([b[1].size for b in boxes])]).astype(np.int64)
    n, eps, theta = int(off[-1]), 1e-3, 0.7
    pos = torch.from_numpy(np.concatenate([b[0] for b in boxes], axis=1).reshape(-1)).cuda()
    mass = torch.from_numpy(np.concatenate([b[1] for b in boxes])).cuda()
    flags = np.zeros(n, np.uint8)
    for lo, hi in zip(off[:-1], off[1:]):  # runs of active particles, the same in equal boxes
        flags[lo:hi] = (np.arange(hi - lo) // 50) % every == 0
    many, one = binding.Context(0, bucket=4, group=16), binding.Context(0, bucket=4, group=16)
    try:
        acc, pot = torch.zeros(3 * n, device="cuda:0"), torch.zeros(n, device="cuda:0")
        many.compute_forces_batch(pos, mass, off, eps, theta, acc, pot, torch.from_numpy(flags).cuda())
        torch.cuda.synchronize()
        assert many.stats()["n_cells"] >= ORDERED and int((many.export_walk_levels()[:, 0] > 0).sum()) > 8
        acc = acc.view(3, n)
        for b in (0, 1, 13, 100, 161, 200, 239):
            lo, hi = int(off[b]), int(off[b + 1])
            a1, p1 = torch.zeros(3 * (hi - lo), device="cuda:0"), torch.zeros(hi - lo, device="cuda:0")
            one.compute_forces(torch.from_numpy(boxes[b][0].reshape(-1).copy()).cuda(), torch.from_numpy(boxes[b][1]).cuda(),
                               eps, theta, a1, p1, torch.from_numpy(flags[lo:hi].copy()).cuda())
            torch.cuda.synchronize()
            assert torch.equal(acc[:, lo:hi], a1.view(3, -1)) and torch.equal(pot[lo:hi], p1), b
    finally:
        many.close()
        one.close()
