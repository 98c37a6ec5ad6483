"""Group local expansions against the oracle's, for groups at every distance from the walk levels whose
cells are evaluated (every fourth) and down chains of many of them.

The oracle re-expands every ancestor's terms to the group in FP64; the GPU goes down step by step in
FP32.  The acceleration the expansion gives at the group's particles may differ by FP32 rounding of
the terms, a few 1e-7 each of the field they sum to; the bounds are the full-size test's (2e-5 rms and
2e-3 at worst of the particle's total, for particles where large terms cancel)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1609_08621_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def _nested(n, seed):
    """Points whose density rises towards a corner by octaves: groups on many consecutive levels."""
    rng = np.random.default_rng(seed)
    r = 2.0 ** -rng.integers(0, 16, n)
    return rng.random((3, n)) * r * 0.999, np.full(n, 1.0 / n, np.float32)


@pytest.mark.parametrize("n,kind", [(40, "plummer"), (65, "plummer"), (300, "plummer"), (6000, "plummer"),
                                    (4000, "nested")])
def test_group_expansions_match_the_oracle(n, kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pos, mass = _nested(n, 3) if kind == "nested" else synth.clustered_plummer(n, 11)
    eps, theta = 1e-4, 0.7
    ctx = binding.Context(0, bucket=8, group=16)
    try:
        acc = torch.zeros(3 * n, dtype=torch.float32, device="cuda:0")
        ctx.compute_forces(torch.from_numpy(pos.reshape(-1).copy()).cuda(), torch.from_numpy(mass).cuda(), eps, theta, acc)
        torch.cuda.synchronize()
        g = ctx.export_cells()
        gcell, gL = ctx.export_locals()
        levels = int((ctx.export_walk_levels()[:, 0] > 0).sum())
    finally:
        ctx.close()
    if kind == "nested":
        assert levels > 20
    orc = oracle.FMM(pos, mass, eps, theta, bucket=8, group=16)
    o, (ocell, oL), perm = orc.cells(), orc.groups(), orc.perm()
    scale = np.linalg.norm(orc.forces()[0], axis=0)
    loc_idx, _ = binding.fmm_multi_index()
    gL = gL[:, [int(np.where((loc_idx == m).all(axis=1))[0][0]) for m in oracle.multi_index()]]
    okey = {(int(o["first"][c]), int(o["count"][c])): i for i, c in enumerate(ocell)}
    assert len(okey) == len(gcell)
    errs = []
    for i, c in enumerate(gcell):
        first, count = int(g["first"][c]), int(g["count"][c])
        j = okey[first, count]
        for q in range(first, first + count):
            p = int(perm[q])
            u = pos[:, p] - o["com"][ocell[j]]
            ag, _ = oracle.l2p(gL[i].astype(np.float64), u)
            ao, _ = oracle.l2p(oL[j], u)
            errs.append(np.linalg.norm(np.asarray(ag) - np.asarray(ao)) / scale[p])
    errs = np.array(errs)
    assert errs.size == n and np.sqrt(np.mean(errs ** 2)) <= 2e-5 and errs.max() <= 2e-3
