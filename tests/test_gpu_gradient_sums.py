"""How the gradient of the learned criterion's network adds its rows: 64 at a time, each 64 in the order of its
rows, and those sums one after another in FP32, as training runs of few rows per step always had them.  An
order or a rounding of its own in the last addition changes the last bit of many gradients, and Adam's
normalised step and the ReLU's kinks carry that into the weights, so it is held to the bit.

Beyond 152 blocks of 64 rows a block takes several of them and goes on with the sums that it has.  Against
the network in FP64, every FP32 addition is off by 6e-8 of the partial sum at most; with at most 64 x 4
rows to a block and 152 blocks behind one another that is 256 + 152 additions, whose errors of random sign
add up to 6e-8 sqrt(408) = 1.2e-6 of the terms' absolute sum; terms that cancel leave a gradient of about
1/sqrt(rows) of it, 1/100 and more here, so 1.2e-4 in norm with room for a factor of about one, rounded up to
2e-4."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as omlp
from paper_1609_08621_gb300 import binding

pytestmark = pytest.mark.gpu

ROWS, BLOCKS = 64, 152  # rows per block and turn, blocks of a gradient


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(6)
    flat = np.zeros(omlp.N_PARAMS)
    flat[:omlp.N_WEIGHTS] = 0.25 * rng.standard_normal(omlp.N_WEIGHTS)
    p = omlp.unpack(flat)
    p["mean"][:] = rng.standard_normal(8)
    p["inv_std"][:] = 0.5 + rng.random(8)
    c = binding.Context(0)
    c.params = omlp.pack(p).astype(np.float32)
    c.mlp_load(c.params)
    yield c
    c.close()


def _rows(n, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n, 8)).astype(np.float32), rng.standard_normal(n).astype(np.float32)


# powers of two, so that the mean over 64 rows and the mean over all differ by an exact factor
@pytest.mark.parametrize("n", [64, 128, 256, 1024, 8192])
def test_blocks_are_added_one_after_another(ctx, n):
    f, y = _rows(n, n)
    f, y = torch.from_numpy(f).cuda(), torch.from_numpy(y).cuda()
    whole, _ = ctx.mlp_gradient(f, y)
    want = np.zeros_like(whole)
    for k in range(0, n, ROWS):
        part, _ = ctx.mlp_gradient(f[k:k + ROWS].contiguous(), y[k:k + ROWS].contiguous())
        want = want + part * np.float32(ROWS / n)
    assert whole.dtype == want.dtype == np.float32
    assert np.array_equal(whole, want)


@pytest.mark.parametrize("n", [ROWS * BLOCKS, ROWS * BLOCKS + 1, 3 * ROWS * BLOCKS + 37])
def test_blocks_of_several_turns(ctx, n):
    f, y = _rows(n, n)
    g, loss = ctx.mlp_gradient(torch.from_numpy(f).cuda(), torch.from_numpy(y).cuda())
    p64 = ctx.params.astype(np.float64)
    want = omlp.grad(p64, f.astype(np.float64), y.astype(np.float64))
    assert np.linalg.norm(g - want) <= 2e-4 * np.linalg.norm(want)
    # the loss is added row by row in FP32: n roundings of 6e-8 of the sum at most
    assert loss == pytest.approx(omlp.loss(p64, f, y), rel=6e-8 * n + 1e-5)


def test_an_infinite_gradient_stays_infinite(ctx):
    f, y = _rows(128, 3)
    y[5] = 3e38  # its error times a weight's input overflows; no sum of opposite infinities
    y[6:] = 0.0
    g, _ = ctx.mlp_gradient(torch.from_numpy(f).cuda() * 1e3, torch.from_numpy(y).cuda())
    assert np.isinf(g).any() and not np.isnan(g).any()
