"""A large walk keeps its sinks in tree order, which takes two more launches per level, whatever the share of
cells to particles and whatever the context has solved before.  Seen from the launch counts of one set of
particles in buckets of 4 (3.5 million cells, ordered) and of 16 (0.9 million, not): apart from those
launches a level costs one, and every fourth level one for the local expansions.  The forces are those of
each box alone, whose walk is not ordered, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu

BOXES, EACH = 50, 100_000


def _solve(ctx, pos, mass, off):
    n = mass.numel()
    acc, pot = torch.zeros(3 * n, device="cuda:0"), torch.zeros(n, device="cuda:0")
    for _ in range(2):  # the first may walk again with larger lists
        ctx.compute_forces_batch(pos, mass, off, 1e-3, 0.9, acc, pot)
    torch.cuda.synchronize()
    st = ctx.stats()
    assert st["retries"] == 0
    # one launch for every level down to the deepest cell, walked or not
    parent, levels = ctx.export_cells()["parent"], 0
    up = parent
    while up.size:
        up = parent[up[up >= 0]]
        levels += 1
    return acc, pot, st["n_cells"], levels, st["n_launches"] - levels - (levels + 3) // 4


@pytest.mark.parametrize("larger_before", [False, True])
def test_order_does_not_depend_on_scratch(larger_before):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda:0").manual_seed(11)
    n = BOXES * EACH
    boxes = [torch.rand(3, EACH, generator=g, device="cuda:0", dtype=torch.float64) for _ in range(BOXES)]
    off = np.arange(BOXES + 1, dtype=np.int64) * EACH
    pos = torch.cat(boxes, 1).contiguous().view(-1)
    mass = torch.full((n,), 1.0 / EACH, device="cuda:0")
    small, large = binding.Context(0, bucket=4, group=16), binding.Context(0, bucket=16, group=16)
    try:
        if larger_before:  # scratch of a larger tree on the same context
            k = 12_000_000
            p = torch.rand(3 * k, generator=g, device="cuda:0", dtype=torch.float64)
            small.build_tree(p, torch.full((k,), 1.0 / k, device="cuda:0"))
        acc, pot, cells, levels, launches = _solve(small, pos, mass, off)
        _, _, few, _, fewer = _solve(large, pos, mass, off)
        assert cells >= 3_000_000 and 4096 < few < 1 << 20  # more than one tile to scan, in both
        assert launches == fewer + 2 * levels
        for b in (0, 7, BOXES - 1):
            lo, hi = int(off[b]), int(off[b + 1])
            a1, p1 = torch.zeros(3 * EACH, device="cuda:0"), torch.zeros(EACH, device="cuda:0")
            small.compute_forces(boxes[b].view(-1), mass[lo:hi].contiguous(), 1e-3, 0.9, a1, p1)
            torch.cuda.synchronize()
            assert torch.equal(acc.view(3, -1)[:, lo:hi], a1.view(3, -1)) and torch.equal(pot[lo:hi], p1), b
    finally:
        small.close()
        large.close()
