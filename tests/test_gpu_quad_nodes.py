"""An odd number of quadrature nodes: the plan's complex tables follow its real ones in one
allocation and must stay on 16-byte boundaries."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf
from paper_1801_05977_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# both node numbers resolve the integrands of these grids to rounding
@pytest.mark.parametrize("dim,precision,tol", [(3, gf.GF_FP64, 1e-11), (3, gf.GF_FP32_SPLIT, 5e-6), (2, gf.GF_FP64, 1e-11)])
def test_odd_quad_nodes(dim, precision, tol):
    if dim == 3:
        x = torch.from_numpy(W.targets_3d(500, seed=5)).cuda()
        args = (3, 2.5, (0.1, 0.3), (16, 16, 16))
    else:
        x = torch.from_numpy(np.random.default_rng(5).uniform(-0.5, 0.5, (500, 2))).cuda()
        args = (2, 1.3, (0.2,), (32, 32))
    out = []
    for nodes in (64, 65):
        p = gf.Plan(*args, precision=precision, quad_nodes=nodes)
        out.append(p.eval_points(x, gf.GF_OUT_GD if dim == 3 else gf.GF_OUT_G).cpu().numpy())
        p.close()
    assert np.abs(out[1] - out[0]).max() < tol * np.abs(out[0]).max()
