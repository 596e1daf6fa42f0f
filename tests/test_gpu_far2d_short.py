"""2D far lists on both sides of the line (2048 targets; more where c is small) between a warp per target and the
table kernel: the same targets give the same values on either route, for all outputs and precisions, few and many
propagating indices, a small c (runs beyond the table, several lanes a target), a large alpha."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(gf.GF_FP64, 1e-12), (gf.GF_FP32_SPLIT, 1e-6)])
@pytest.mark.parametrize("n,k,k2,alpha,c,zmax", [(2049, 1.3, 2.1, 0.2, 0.6, 1.0), (2049, 0.15, 0.3, 0.45, 0.6, 90.0),
                                                 (2049, 40.3, 41.7, 0.1, 0.6, 2.0), (14001, 2.5, 1.1, -0.37, 0.05, 0.3),
                                                 (36001, 1.3, 2.1, 0.2, 0.02, 0.1), (2049, 1.3, 2.1, -37.8, 0.6, 1.0)])
def test_both_routes(precision, tol, n, k, k2, alpha, c, zmax):
    rng = np.random.default_rng(1)
    x = np.c_[rng.uniform(-9.0, 9.0, n), rng.uniform(c, zmax, n) * rng.choice([-1.0, 1.0], n)]
    x[0, 1] = np.nextafter(c, 1.0)
    xd = torch.from_numpy(x).cuda()
    for kind, which in ((gf.GF_HELMHOLTZ, gf.GF_OUT_G), (gf.GF_DERIV2D, gf.GF_OUT_GRAD), (gf.GF_DERIV2D, gf.GF_OUT_HESSDIFF)):
        p = gf.Plan(2, k, (alpha,), (16, 16), c=c, precision=precision, kind=kind, k2=k2 if kind == gf.GF_DERIV2D else 0.0)
        long = p.eval_points(xd, which)
        short = torch.cat([p.eval_points(v, which) for v in xd.split(2048)])
        p.close()
        assert float(((long - short).abs().amax(0) / short.abs().amax(0)).max()) < tol, which
