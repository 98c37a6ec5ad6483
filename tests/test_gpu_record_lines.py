"""Results of large solves go through records where they cost less than direct stores: from 11 * 2^19 particles on,
with at least a quarter of them active.  Which way a solve took is seen from its launch count (the records'
split is one more); both ways give the same bits, so a batch that takes the records is compared with its
boxes solved alone, which do not, and particles that are not active keep what the caller's arrays held."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu

LINE = 11 << 19
MARK = 7.0


def _box(n, seed):
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    pos = torch.rand(3 * n, generator=g, device="cuda:0", dtype=torch.float64)
    return pos, torch.full((n,), 1.0 / n, device="cuda:0"), torch.rand(n, generator=g, device="cuda:0")


def _results(n):
    return torch.full((3 * n,), MARK, device="cuda:0"), torch.full((n,), MARK, device="cuda:0")


@pytest.fixture
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = binding.Context(0, accumulate=1)
    yield c
    c.close()


@pytest.mark.parametrize("n,records", [(LINE, True), (LINE - 1, False), (1 << 22, False)])
def test_line(ctx, n, records):
    pos, mass, u = _box(n, n)
    quarter = (torch.arange(n, device="cuda:0") % 4 == 0).to(torch.uint8)
    assert 4 * int(quarter.sum()) >= n
    fewer = quarter.clone()
    fewer[:8] = 0  # less than a quarter
    assert 4 * int(fewer.sum()) < n
    launches = []
    for flags in (quarter, fewer):
        acc, pot = _results(n)
        for _ in range(2):  # the first may walk again with larger lists
            ctx.compute_forces(pos, mass, 1e-3, 0.95, acc, pot, flags)
        torch.cuda.synchronize()
        st = ctx.stats()
        assert st["retries"] == 0
        launches.append(st["n_launches"])
        on = flags.bool()
        acc = acc.view(3, n)
        assert bool((acc[:, ~on] == MARK).all()) and bool((pot[~on] == MARK).all())
        assert not bool((acc[:, on] == MARK).all(0).any()) and bool(torch.isfinite(acc).all())
    assert launches[0] - launches[1] == (1 if records else 0)


@pytest.mark.parametrize("pot", [True, False])
def test_batch_by_records_equals_boxes_by_direct_stores(ctx, pot):
    # unequal boxes, an empty one, tiny neighbours, one with nothing active; more than a quarter active in all
    sizes = [1_000_000, 0, 3, 2, 1_500_001, 17, 1_200_000, 900_000, 1_400_000, 1]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    assert n >= LINE
    parts = [_box(max(k, 1), 50 + i) for i, k in enumerate(sizes)]
    pos3 = torch.cat([p.view(3, -1)[:, :k] for (p, _, _), k in zip(parts, sizes)], 1).contiguous()
    mass = torch.cat([m[:k] for (_, m, _), k in zip(parts, sizes)])
    flags = torch.cat([(u[:k] < 0.4) for (_, _, u), k in zip(parts, sizes)]).to(torch.uint8)
    flags[int(off[6]):int(off[7])] = 0
    for b in (2, 3, 9):
        flags[int(off[b])] = 1
    assert 4 * int(flags.sum()) >= n
    acc, p = _results(n)
    ctx.compute_forces_batch(pos3.view(-1), mass, off, 1e-3, 0.9, acc, p if pot else None, flags)
    torch.cuda.synchronize()
    acc = acc.view(3, n)
    if not pot:
        assert bool((p == MARK).all())
    for b, k in enumerate(sizes):
        if k == 0:
            continue
        lo, hi = int(off[b]), int(off[b + 1])
        a1, p1 = _results(k)
        f = flags[lo:hi].contiguous()
        if int(f.sum()):
            ctx.compute_forces(pos3[:, lo:hi].contiguous().view(-1), mass[lo:hi].contiguous(), 1e-3, 0.9, a1, p1, f)
        torch.cuda.synchronize()
        assert torch.equal(acc[:, lo:hi], a1.view(3, k)), b
        assert not pot or torch.equal(p[lo:hi], p1), b


def test_replay_with_fewer_active_than_at_the_capture(ctx):
    # the way is chosen at the capture; flags that fall under a quarter afterwards still give the same results
    pos, mass, u = _box(LINE, 9)
    flags = (u < 0.3).to(torch.uint8)
    few = (u < 0.05).to(torch.uint8)
    ctx.set_graphs(True)
    acc, pot = _results(LINE)
    for _ in range(3):
        ctx.compute_forces(pos, mass, 1e-3, 0.95, acc, pot, flags)
    torch.cuda.synchronize()
    before = ctx.graph_info()
    first, on = acc.view(3, LINE).clone(), few.bool()
    flags.copy_(few)
    acc.fill_(MARK)
    pot.fill_(MARK)
    ctx.compute_forces(pos, mass, 1e-3, 0.95, acc, pot, flags)
    torch.cuda.synchronize()
    assert ctx.graph_info() != before  # replayed
    a = acc.view(3, LINE)
    assert bool((a[:, ~on] == MARK).all()) and bool((pot[~on] == MARK).all())
    eager = binding.Context(0, accumulate=1)
    try:
        e, q = _results(LINE)
        eager.compute_forces(pos, mass, 1e-3, 0.95, e, q, few)
        torch.cuda.synchronize()
        assert 4 * int(few.sum()) < LINE and torch.equal(acc, e) and torch.equal(pot, q)
    finally:
        eager.close()
    # beside the solve with more active sinks: the same lists, sums split over lanes by the sinks in them
    d = (a[:, on] - first[:, on]).norm(dim=0) / first[:, on].norm(dim=0)
    assert float(d.square().mean().sqrt()) <= 1e-5
