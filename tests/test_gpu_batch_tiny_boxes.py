"""Boxes of a few particles beside one another in one solve: neighbours of together no more than a bucket are
still boxes of their own, and every box's forces are those of the box alone, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,bucket,every", [
    ([1, 2], 16, 1),                                       # the whole input is less than a bucket
    ([1, 1, 1, 1, 1], 16, 1),
    ([2, 3, 0, 1, 15, 1, 16, 1, 17, 1, 1, 0, 0, 2], 16, 1),  # empty boxes and bucket-sized ones between
    ([1, 2, 3, 2000, 1, 4, 64, 2, 3000, 5, 6, 7], 16, 1),
    ([1, 2, 3, 2000, 1, 4, 64, 2, 3000, 5, 6, 7], 4, 3),     # a part of the particles active
    ([1 + i % 5 for i in range(256)], 8, 1),               # the most boxes a call takes
])
def test_each_box_as_alone(sizes, bucket, every):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    boxes = [synth.clustered_plummer(max(k, 1), 700 + i) for i, k in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, eps, theta = int(off[-1]), 1e-3, 0.7
    pos = np.concatenate([b[0][:, :k] for b, k in zip(boxes, sizes)], axis=1)
    mass = np.concatenate([b[1][:k] for b, k in zip(boxes, sizes)])
    flags = (np.arange(n) % every == 0).astype(np.uint8)
    ctx = binding.Context(0, bucket=bucket, group=max(bucket, 16))

    def solve(p, m, f, offsets=None):
        k = m.size
        acc, pot = torch.full((3 * k,), float("nan"), device="cuda:0"), torch.full((k,), float("nan"), device="cuda:0")
        args = [torch.from_numpy(np.ascontiguousarray(p).reshape(-1)).cuda(), torch.from_numpy(np.ascontiguousarray(m)).cuda()]
        f = torch.from_numpy(np.ascontiguousarray(f)).cuda()
        if offsets is None:
            ctx.compute_forces(*args, eps, theta, acc, pot, f)
        else:
            ctx.compute_forces_batch(*args, offsets, eps, theta, acc, pot, f)
        torch.cuda.synchronize()
        return acc.cpu().numpy().reshape(3, k), pot.cpu().numpy()

    try:
        acc, pot = solve(pos, mass, flags, off)
        on = flags.astype(bool)
        assert np.isfinite(acc[:, on]).all() and np.isfinite(pot[on]).all()
        assert np.isnan(acc[:, ~on]).all() and np.isnan(pot[~on]).all()
        for b, (lo, hi) in enumerate(zip(off[:-1], off[1:])):
            if not on[lo:hi].any():
                continue
            a1, p1 = solve(pos[:, lo:hi], mass[lo:hi], flags[lo:hi])
            assert np.array_equal(acc[:, lo:hi], a1, equal_nan=True) and np.array_equal(pot[lo:hi], p1, equal_nan=True), b
    finally:
        ctx.close()
