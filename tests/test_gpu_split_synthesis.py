"""The split plans' first synthesis pass (tiles of columns in float, single columns in double)
against the double-precision plans: the smallest and longest last axes (radix-2 first stage or
not, tiles of 8, 16 and 32 columns), few and many quadrature nodes, wave numbers that put no, a
few or all columns of the grid among the double ones, a Wood anomaly, a large alpha, one and
seven fields."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf
from paper_1801_05977_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [  # k, alpha, M, quadrature nodes (0: automatic)
    (2.5, (0.1, 0.3), (8, 8, 8), 0),
    (2.5, (0.1, 0.3), (8, 16, 16), 13),
    (0.3, (0.5, -0.2), (32, 16, 64), 0),
    (1.42, (0.3, 1.0), (16, 32, 32), 1024),   # |alpha_n| within 2 per cent of k
    (14.3, (0.1, 0.2), (16, 16, 128), 0),     # every column double
    (3.7, (5.3, -40.25), (64, 32, 256), 0),   # the double columns at one edge, and off the grid
    (2.5, (0.1, 0.3), (8, 8, 1024), 0),
]


# float coefficients (a few 2^-24 each), a transform of up to 1024 x 64 x 32 terms (log2 of the
# terms roundings of 2^-24 along each chain) and a float stencil: 5e-6 of the largest value
@pytest.mark.parametrize("kind", [gf.GF_HELMHOLTZ, gf.GF_MAXWELL])
@pytest.mark.parametrize("k,alpha,M,nodes", CASES)
def test_split_synthesis_against_double(k, alpha, M, nodes, kind):
    x = W.targets_3d(4000, seed=3)
    x[:, 2] = np.random.default_rng(4).uniform(-0.6, 0.6, len(x))
    x = torch.from_numpy(x).cuda()
    which = gf.GF_OUT_GD if kind == gf.GF_HELMHOLTZ else gf.GF_OUT_MAXWELL7
    out = []
    for precision in (gf.GF_FP64, gf.GF_FP32_SPLIT):
        p = gf.Plan(3, k, alpha, M, precision=precision, kind=kind, quad_nodes=nodes)
        out.append(p.eval_points(x, which).cpu().numpy())
        p.close()
    err = np.abs(out[1] - out[0]).max(axis=0) / np.abs(out[0]).max(axis=0)
    assert err.max() < 5e-6, err
