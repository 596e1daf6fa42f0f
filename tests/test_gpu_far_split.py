"""The split plans' Helmholtz far series on long lists (two targets a lane; from 786432 targets on
the matrix products) against the same targets in short calls (one target a lane, row slabs): ragged lists
with an odd number of chunks, no, some and many propagating indices, and a batched sweep long enough for
two targets a lane against its pairs' own plans."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu

# both forms sum about 3000 float terms per target with the same weights and phases; their roundings
# differ by a few 2^-24 of the largest row each
TOL = 5e-6


def far_cloud(n, seed):
    rng = np.random.default_rng(seed)
    x = np.empty((n, 3))
    x[:, :2] = rng.uniform(-9.0, 9.0, (n, 2))
    x[:, 2] = rng.uniform(0.6 + 1e-9, 1.0, n) * rng.choice([-1.0, 1.0], n)
    return torch.from_numpy(x).cuda()


@pytest.mark.parametrize("k,n", [(0.31, 130000), (2.5, 400015), (5.2, 200033), (2.5, 790001)])
def test_long_lists(k, n):
    x = far_cloud(n, n)
    p = gf.Plan(3, k, (0.45, 0.3), (16, 16, 16), precision=gf.GF_FP32_SPLIT)
    long = p.eval_points(x, gf.GF_OUT_GD)
    short = torch.cat([p.eval_points(c, gf.GF_OUT_GD) for c in x.split(20000)])
    p.close()
    assert torch.isfinite(torch.view_as_real(long)).all()
    assert float((long - short).abs().max() / short.abs().max()) < TOL


def test_long_sweep():
    k, al = np.array([2.5, 0.4, 4.3]), np.array([[0.1, 0.3], [0.45, 0.1], [-0.2, 0.4]])
    M = np.full((3, 3), 16)
    off = np.array([0, 150017, 150017, 400000], dtype=np.int64)
    x = far_cloud(int(off[-1]), 3)
    b = gf.Batch(k, al, M, precision=gf.GF_FP32_SPLIT)
    out = torch.empty((len(x), 1), dtype=torch.complex64, device="cuda")
    b.eval_points_into(x, off, out, gf.GF_OUT_GD)
    for i in (0, 2):
        p = gf.Plan(3, k[i], al[i], M[i], precision=gf.GF_FP32_SPLIT)
        ref = torch.cat([p.eval_points(c, gf.GF_OUT_GD) for c in x[off[i]:off[i + 1]].split(20000)])
        p.close()
        assert float((out[off[i]:off[i + 1]] - ref).abs().max() / ref.abs().max()) < TOL, i
    b.close()
