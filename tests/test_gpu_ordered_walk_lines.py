"""From how many cells a walk keeps its sinks in tree order: a box of 1.3 million cells does with the learned
criterion, not with the fixed one, whose shorter queues lose more to the two launches per level than
they gain below 2.6 million.  Seen from the launch counts beside a box of 0.9 million cells, which does not."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as omlp
from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu


def _network():
    """Untrained weights: only launches are counted."""
    rng = np.random.default_rng(4)
    flat = np.zeros(omlp.N_PARAMS)
    flat[:omlp.N_WEIGHTS] = 0.25 * rng.standard_normal(omlp.N_WEIGHTS)
    p = omlp.unpack(flat)
    p["inv_std"][:] = 1.0
    return omlp.pack(p).astype(np.float32)


def _launches(n, criterion):
    """(cells, levels, launches but for those of the levels) of a solve with a few particles active"""
    g = torch.Generator(device="cuda:0").manual_seed(n)
    pos = torch.rand(3 * n, generator=g, device="cuda:0", dtype=torch.float64)
    mass = torch.full((n,), 1.0 / n, device="cuda:0")
    active = (torch.arange(n, device="cuda:0") % 1000 == 0).to(torch.uint8)
    acc, pot = torch.ones(3 * n, device="cuda:0"), torch.zeros(n, device="cuda:0")
    ctx = binding.Context(0)
    try:
        if criterion:
            ctx.mlp_load(_network())
            ctx.set_params(criterion=1, mlp_tau=-3.5)
        for _ in range(2):  # the first may walk again with larger lists
            ctx.compute_forces(pos, mass, 1e-3, 0.9, acc, pot, active)
        torch.cuda.synchronize()
        st = ctx.stats()
        assert st["retries"] == 0
        parent, levels = ctx.export_cells()["parent"], 0
        up = parent
        while up.size:
            up = parent[up[up >= 0]]
            levels += 1
        return st["n_cells"], levels, st["n_launches"] - levels - (levels + 3) // 4
    finally:
        ctx.close()


@pytest.mark.parametrize("criterion", [0, 1])
def test_lines_of_the_two_criteria(criterion):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    few, _, below = _launches(5_000_000, criterion)
    cells, levels, above = _launches(7_000_000, criterion)
    assert few < 1 << 20 <= cells < 5 << 19
    assert above == below + (2 * levels if criterion else 0)
