"""The training pass at the sizes where its tiling can go wrong: ragged last tiles of
128 rows, row ranges of unequal length in the split weight gradients, more tiles
than CTAs, and inputs that are only 4-byte aligned."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as R
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


def samples(n, seed):
    rng = np.random.default_rng(seed)
    inp = np.column_stack([rng.uniform(-np.pi, np.pi, (n, 2)), rng.uniform(-0.6, 0.6, n),
                           rng.uniform(-0.5, 0.5, (n, 2)), rng.uniform(1, 4, n)]).astype(np.float32)
    return inp, rng.standard_normal((n, 2)).astype(np.float32)


def bf16_round(a):
    return torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16).float().numpy()


@pytest.mark.parametrize("n", [65, 128, 1000, 2049])
def test_gradients_at_ragged_sizes(n):
    """Against the FP64 reference with bf16-rounded weights, 6e-2 of each layer's largest
    gradient (the bf16 activations' rounding, as for the full-tile test); the same bits twice."""
    mlp = gf.MLP(seed=4)
    Ws, bs = R.unpack(mlp.get_params())
    pr = R.pack([bf16_round(W) for W in Ws[:4]] + [Ws[4]], bs)
    inp, tgt = samples(n, n)
    x, t = torch.from_numpy(inp).cuda(), torch.from_numpy(tgt).cuda()
    g, loss = mlp.gradients(x, t)
    lref, gref = R.loss_and_grad(pr, inp.astype(np.float64), tgt.astype(np.float64))
    assert abs(loss - lref) < 2e-2 * lref
    off = 0
    for l in range(5):
        m = R.DIMS[l + 1] * R.DIMS[l] + R.DIMS[l + 1]
        assert np.abs(g[off:off + m] - gref[off:off + m]).max() < 6e-2 * np.abs(gref[off:off + m]).max(), l
        off += m
    g2, loss2 = mlp.gradients(x, t)
    assert np.array_equal(g, g2) and loss == loss2
    mlp.close()


@pytest.mark.parametrize("n", [1024, 32768])
def test_gradient_of_a_batch_is_the_mean_of_its_halves(n):
    """1/n is a power of two in all three calls, so every bf16 rounding is the same and only
    the order of the float sums differs: about 2^-24 sqrt(65536) = 1.5e-5 of the terms' size,
    3e-5 of the layer's largest gradient asked (65536 rows: more tiles than SMs)."""
    mlp = gf.MLP(seed=6)
    inp, tgt = samples(2 * n, 9)
    x, t = torch.from_numpy(inp).cuda(), torch.from_numpy(tgt).cuda()
    g, _ = mlp.gradients(x, t)
    a, _ = mlp.gradients(x[:n], t[:n])
    b, _ = mlp.gradients(x[n:], t[n:])
    h = 0.5 * (a.astype(np.float64) + b)
    off = 0
    for l in range(5):
        m = R.DIMS[l + 1] * R.DIMS[l] + R.DIMS[l + 1]
        assert np.abs(g[off:off + m] - h[off:off + m]).max() < 3e-5 * np.abs(h[off:off + m]).max(), l
        off += m
    assert mlp.error_word() == 0
    mlp.close()


def test_unaligned_inputs():
    """Inputs at an odd float offset of a larger buffer give the bits of the aligned ones."""
    mlp = gf.MLP(seed=7)
    inp, tgt = samples(300, 3)
    x, t = torch.from_numpy(inp).cuda(), torch.from_numpy(tgt).cuda()
    bx = torch.zeros(300 * 6 + 1, device="cuda")
    bx[1:] = x.reshape(-1)
    bt = torch.zeros(300 * 2 + 1, device="cuda")
    bt[1:] = t.reshape(-1)
    g, loss = mlp.gradients(x, t)
    g1, loss1 = mlp.gradients(bx[1:].view(300, 6), bt[1:].view(300, 2))
    assert np.array_equal(g, g1) and loss == loss1
    assert torch.equal(mlp.forward(x), mlp.forward(bx[1:].view(300, 6)))
    mlp.close()
