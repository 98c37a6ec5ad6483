"""Solves of 2^22 particles and more write their results as records and split them afterwards where at
least a quarter of the particles is active; below either line they write the caller's arrays directly.
Both must leave inactive particles alone, skip a NULL potential, and give the same bits: the solve with
every particle active against one whose inactive flags keep the direct stores, on a box just past the
line, and the same box one particle short of it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu
LINE = 1 << 22


def _solve(ctx, pos, mass, active, pot=True):
    n = mass.numel()
    acc = torch.full((3 * n,), 7.0, device="cuda:0")
    p = torch.full((n,), 7.0, device="cuda:0") if pot else None
    ctx.compute_forces(pos, mass, 1e-3, 0.9, acc, p, active)
    torch.cuda.synchronize()
    return acc.view(3, n), p


@pytest.mark.parametrize("n,share,accumulate", [(LINE, 0.5, 1), (LINE + 77, 0.26, 0), (LINE - 1, 0.5, 1)])
def test_records_and_direct_stores_agree(n, share, accumulate):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = torch.Generator(device="cuda:0").manual_seed(n)
    pos = torch.rand(3 * n, generator=g, device="cuda:0", dtype=torch.float64)
    mass = torch.full((n,), 1.0 / n, device="cuda:0")
    many = (torch.rand(n, generator=g, device="cuda:0") < share).to(torch.uint8)
    few = many * (torch.rand(n, generator=g, device="cuda:0") < 0.3).to(torch.uint8)  # under a quarter: direct
    assert 4 * int(many.sum()) >= n > 4 * int(few.sum())
    ctx = binding.Context(0, accumulate=accumulate)
    try:
        a, p = _solve(ctx, pos, mass, many)
        d, q = _solve(ctx, pos, mass, few)
        on, both = many.bool(), few.bool()
        assert bool((a[:, ~on] == 7.0).all()) and bool((p[~on] == 7.0).all())
        assert bool((d[:, ~both] == 7.0).all()) and bool((q[~both] == 7.0).all())
        assert not bool((a[:, on] == 7.0).all(0).any())
        # the sinks of both solves: the same lists, sums split over lanes by the sinks beside them
        diff = (a[:, both] - d[:, both]).norm(dim=0) / a[:, both].norm(dim=0)
        assert float(diff.max()) <= 1e-3 and float(diff.square().mean().sqrt()) <= 1e-5
        b, none = _solve(ctx, pos, mass, many, pot=False)
        assert none is None and torch.equal(a, b)
    finally:
        ctx.close()
