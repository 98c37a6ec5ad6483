"""The M2L pass takes the walk's flat list in chunks of 32 sources, copied a chunk ahead, and carries a
sink whose list goes on into the next chunk.  Against the oracle's group expansions, with lists from a
few sources per sink to several chunks of them.

Bounds as for any FP32 group expansion against the FP64 one: rounding of the terms, a few 1e-7 each of
the field that they sum to; 2e-5 rms and 2e-3 at worst of the particle's total acceleration."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1609_08621_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,theta,bucket,group", [(90, 0.9, 2, 4), (1500, 0.45, 4, 8), (5000, 0.6, 2, 2), (9000, 0.9, 16, 64)])
def test_chunks_of_multipole_sources(n, theta, bucket, group):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pos, mass = synth.clustered_plummer(n, 17)
    eps = 1e-4
    ctx = binding.Context(0, bucket=bucket, group=group)
    try:
        acc = torch.zeros(3 * n, dtype=torch.float32, device="cuda:0")
        ctx.compute_forces(torch.from_numpy(pos.reshape(-1).copy()).cuda(), torch.from_numpy(mass).cuda(), eps, theta, acc)
        torch.cuda.synchronize()
        g = ctx.export_cells()
        gcell, gL = ctx.export_locals()
        assert ctx.stats()["n_cc"] > 0
    finally:
        ctx.close()
    orc = oracle.FMM(pos, mass, eps, theta, bucket=bucket, group=group)
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
        for p in map(int, perm[first:first + count]):
            u = pos[:, p] - o["com"][ocell[j]]
            ag, _ = oracle.l2p(gL[i].astype(np.float64), u)
            ao, _ = oracle.l2p(oL[j], u)
            errs.append(np.linalg.norm(np.asarray(ag) - np.asarray(ao)) / scale[p])
    errs = np.array(errs)
    assert errs.size == n and np.sqrt(np.mean(errs ** 2)) <= 2e-5 and errs.max() <= 2e-3
