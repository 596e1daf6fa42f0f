"""The radial transforms' panels (Taylor sums at the panel centres; interpolation for 2 eps > 1): plans
with few and many nodes, small and large eps on both sides of the rule, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu

# eps, c~, nodes: the rule's two sides, one chunk of nodes (128) and several with a remainder
CUTOFFS = [(0.45, 1.0, 0), (0.5, 1.1, 96), (0.505, 1.1, 96), (0.2, 1.0, 200), (0.45, 1.0, 331)]


# as the other double-precision comparisons with the oracle: 1e-10 of each value (floor 1e-6 of the largest)
def rel_err(got, ref):
    scale = np.maximum(np.abs(ref), 1e-6 * np.abs(ref).max(axis=0))
    return float((np.abs(got - ref) / scale).max())


def problem(p, dim, k, al, M):
    i = p.info
    return O.Problem(dim=dim, k=k, alpha=al, M=M, c=i.c, ct=i.c_tilde, eps=i.eps, Q=i.quad_nodes)


@pytest.mark.parametrize("eps,ct,nodes", CUTOFFS)
def test_panels_3d(eps, ct, nodes):
    M, al = (32, 16, 32), (0.1, 0.3)
    rng = np.random.default_rng(2)
    x = np.c_[rng.uniform(-3.1, 3.1, (400, 2)), rng.uniform(-0.6, 0.6, 400)]
    p = gf.Plan(3, 2.5, al, M, quad_nodes=nodes, eps=eps, c_tilde=ct)
    got = p.eval_points(torch.from_numpy(x).cuda(), gf.GF_OUT_GD).cpu().numpy()
    pb = problem(p, 3, 2.5, al, M)
    p.close()
    assert rel_err(got, O.evaluate(pb, O.grid(pb), x, O.OUT_GD)) < 1e-10


@pytest.mark.parametrize("eps,ct,nodes", CUTOFFS)
def test_panels_2d(eps, ct, nodes):
    M, al, k, k2 = (32, 64), (0.2,), 1.3, 2.1
    rng = np.random.default_rng(3)
    x = np.c_[rng.uniform(-3.1, 3.1, 400), rng.uniform(-0.6, 0.6, 400)]
    xd = torch.from_numpy(x).cuda()
    p = gf.Plan(2, k, al, M, quad_nodes=nodes, eps=eps, c_tilde=ct)
    got = p.eval_points(xd, gf.GF_OUT_G).cpu().numpy()
    pb = problem(p, 2, k, al, M)
    p.close()
    G = O.evaluate(pb, O.grid(pb), x, O.OUT_G)
    assert rel_err(got, G) < 1e-10
    p = gf.Plan(2, k, al, M, quad_nodes=nodes, eps=eps, c_tilde=ct, kind=gf.GF_DERIV2D, k2=k2)
    grad, hess = (p.eval_points(xd, w).cpu().numpy() for w in (gf.GF_OUT_GRAD, gf.GF_OUT_HESSDIFF))
    pb = problem(p, 2, k, al, M)
    p.close()
    g = O.grid_deriv2(pb, k2)
    G = O.evaluate(pb, O.grid(pb), x, O.OUT_G)
    assert rel_err(grad, np.concatenate([G, O.evaluate_deriv2(pb, k2, g, x, O.DERIV_GRAD)], axis=1)) < 1e-10
    assert rel_err(hess, O.evaluate_deriv2(pb, k2, g, x, O.DERIV_HYPER)) < 1e-10
