"""The 2D far series at distant targets: propagating indices with |beta_n||x2| from 2^25 on, where the
exponential table's index (discarded for them) no longer fits its integer.  Lists short and long, all
three outputs, both wave numbers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu

K, K2, AL = 1.3, 2.1, 0.2


@pytest.mark.parametrize("n", [7, 6000])
@pytest.mark.parametrize("z", [2.7e7, 1e8, 3.3e9, 7.7e11])
def test_distant(n, z):
    rng = np.random.default_rng(n)
    x = np.c_[rng.uniform(-3.0, 3.0, n), z * rng.uniform(1.0, 1.1, n) * rng.choice([-1.0, 1.0], n)]
    xd = torch.from_numpy(x).cuda()
    ref = slice(0, n, max(1, n // 300))
    p = gf.Plan(2, K, (AL,), (16, 16), kind=gf.GF_DERIV2D, k2=K2)
    grad, hess = (p.eval_points(xd, w).cpu().numpy()[ref] for w in (gf.GF_OUT_GRAD, gf.GF_OUT_HESSDIFF))
    i = p.info
    p.close()
    p = gf.Plan(2, K, (AL,), (16, 16))
    got = p.eval_points(xd, gf.GF_OUT_G).cpu().numpy()[ref]
    p.close()
    pb = O.Problem(dim=2, k=K, alpha=(AL,), M=(16, 16), c=i.c, ct=i.c_tilde, eps=i.eps, Q=i.quad_nodes)
    g = O.grid_deriv2(pb, K2)
    G = O.evaluate(pb, O.grid(pb), x[ref], O.OUT_G)
    # a phase beta |x2| is rounded twice on either side (beta itself by an ulp, the product by half of one):
    # 3 beta |x2| 2^-53 each, beta <= K2
    tol = 6 * K2 * 1.1 * z * 2.0 ** -53
    for a, b in ((got, G), (grad, np.concatenate([G, O.evaluate_deriv2(pb, K2, g, x[ref], O.DERIV_GRAD)], axis=1)),
                 (hess, O.evaluate_deriv2(pb, K2, g, x[ref], O.DERIV_HYPER))):
        assert np.isfinite(a).all()
        assert (np.abs(a - b).max(axis=0) <= tol * np.abs(b).max(axis=0)).all()
