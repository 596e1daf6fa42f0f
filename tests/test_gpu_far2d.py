"""The 2D far series against the oracle: list lengths from one target to more than a CTA takes at once
(one to 32 lanes a target), a small c (more indices than the CTA's table holds), distant targets
(weights beyond the exponential's table), many and no propagating indices, an index next to a Wood anomaly,
a large alpha, both signs of x2, all three outputs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu

CASES = [  # k, k2, alpha, c, n, largest |x2|
    (1.3, 2.1, 0.2, 0.6, 1, 1.0),
    (1.3, 2.1, 0.2, 0.6, 5, 1.0),
    (1.3, 2.1, 0.2, 0.6, 700, 1.0),
    (1.3, 2.1, 0.2, 0.6, 90000, 1.0),
    (2.5, 1.1, -0.37, 0.05, 400, 0.3),
    (0.15, 0.3, 0.45, 0.6, 300, 90.0),
    (40.3, 41.7, 0.1, 0.6, 300, 2.0),
    (1.2001, 1.3, 0.2, 0.6, 300, 2.0),
    (1.3, 2.1, -37.8, 0.6, 300, 1.0),
]


# pointwise, as the other double-precision comparisons with the oracle
def rel_err(got, ref):
    scale = np.maximum(np.abs(ref), 1e-6 * np.abs(ref).max(axis=0))
    return float((np.abs(got - ref) / scale).max())


@pytest.mark.parametrize("k,k2,alpha,c,n,zmax", CASES)
def test_far2d(k, k2, alpha, c, n, zmax):
    rng = np.random.default_rng(n)
    x = np.c_[rng.uniform(-9.0, 9.0, n), rng.uniform(c, zmax, n) * rng.choice([-1.0, 1.0], n)]
    x[0, 1] = np.nextafter(c, 1.0)
    xd = torch.from_numpy(x).cuda()
    ref = slice(0, n, max(1, n // 500))  # the oracle on a part of a long list
    p = gf.Plan(2, k, (alpha,), (16, 16), c=c, kind=gf.GF_DERIV2D, k2=k2)
    grad, hess = (p.eval_points(xd, w).cpu().numpy()[ref] for w in (gf.GF_OUT_GRAD, gf.GF_OUT_HESSDIFF))
    i = p.info
    pb = O.Problem(dim=2, k=k, alpha=(alpha,), M=(16, 16), c=i.c, ct=i.c_tilde, eps=i.eps, Q=i.quad_nodes)
    p.close()
    p = gf.Plan(2, k, (alpha,), (16, 16), c=c)
    got = p.eval_points(xd, gf.GF_OUT_G).cpu().numpy()[ref]
    p.close()
    g = O.grid_deriv2(pb, k2)
    G = O.evaluate(pb, O.grid(pb), x[ref], O.OUT_G)
    assert rel_err(got, G) < 1e-10
    assert rel_err(grad, np.concatenate([G, O.evaluate_deriv2(pb, k2, g, x[ref], O.DERIV_GRAD)], axis=1)) < 1e-10
    assert rel_err(hess, O.evaluate_deriv2(pb, k2, g, x[ref], O.DERIV_HYPER)) < 1e-10
