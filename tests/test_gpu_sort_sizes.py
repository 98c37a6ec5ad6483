"""The stable Morton sort at the sizes where its path changes: one block for up to 8192 keys (1, 2, 4 or
8 per thread), tiles of 2048 keys beyond, tiles that end inside a warp, many equal keys; and the tree
built on it, whose scans take one, two or three launches.  The order must be numpy's stable sort of
the keys, exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1024, 1025, 2048, 2049, 4096, 4097, 8191, 8192, 8193, 10240, 100_003,
                               4_194_305])
def test_order_is_the_stable_sort_of_the_keys(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(n)
    pos = rng.random((3, n))
    pos[:, ::3] = np.floor(pos[:, ::3] * 4) / 4  # a third of the points on 64 places: runs of equal keys
    tpos = torch.from_numpy(pos.reshape(-1).copy()).cuda()
    mass = torch.full((n,), 1.0 / n, dtype=torch.float32, device="cuda:0")
    q = np.floor(pos * 2097152.0).astype(np.uint64)

    def spread(v):
        out = np.zeros_like(v)
        for b in range(21):
            out |= ((v >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b)
        return out

    key = (spread(q[0]) << np.uint64(2)) | (spread(q[1]) << np.uint64(1)) | spread(q[2])
    want = np.argsort(key, kind="stable").astype(np.uint32)
    ctx = binding.Context(0)
    try:
        ctx.build_tree(tpos, mass)
        perm, keys = ctx.export_order(n)
        cells = ctx.export_cells()
    finally:
        ctx.close()
    assert np.array_equal(perm, want) and np.array_equal(keys, key[want])
    leaf = cells["child"][:, 0] < 0  # the buckets partition the sorted particles
    first = np.sort(cells["first"][leaf])
    assert cells["count"][leaf].sum() == n and first[0] == 0 and np.all(cells["count"][leaf] <= 16)
    if n <= binding.STATIC_ORDER_MAX_N:
        k = torch.zeros(n, dtype=torch.int64, device="cuda:0")
        o = torch.zeros(n, dtype=torch.int32, device="cuda:0")
        binding.morton_order_static(tpos, k, o)
        assert np.array_equal(o.cpu().numpy().view(np.uint32), want)
        assert np.array_equal(k.cpu().numpy().view(np.uint64), key[want])
