"""The X' sums of evanescent columns from panels (double 3D plans from 1024 columns on) against the oracle:
the rule's two sides in the columns and in the number of panels (a narrow and a wide transition, the last
too wide), a column next to a Wood anomaly, few and many nodes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


# as the other double-precision comparisons with the oracle: 1e-10 of each value (floor 1e-6 of the largest)
@pytest.mark.parametrize("k,al,M,c,ct,nodes", [
    (2.5, (0.1, 0.3), (32, 32, 16), 0.6, 1.0, 0),
    (2.5, (0.1, 0.3), (32, 16, 16), 0.6, 1.0, 0),
    (1.0005, (0.0, 0.2), (64, 32, 32), 0.6, 1.0, 41),
    (2.5, (0.1, 0.3), (32, 32, 64), 0.5, 1.7, 0),
    (2.5, (0.1, 0.3), (32, 32, 32), 0.3, 3.0, 300),
    (1.4, (-0.3, 0.5), (32, 64, 128), 0.6, 0.92, 0),
])
def test_xprime_panels(k, al, M, c, ct, nodes):
    rng = np.random.default_rng(7)
    x = np.c_[rng.uniform(-3.1, 3.1, (300, 2)), rng.uniform(-c, c, 300)]
    p = gf.Plan(3, k, al, M, c=c, c_tilde=ct, quad_nodes=nodes)
    got = p.eval_points(torch.from_numpy(x).cuda(), gf.GF_OUT_GD).cpu().numpy()
    i = p.info
    p.close()
    pb = O.Problem(dim=3, k=k, alpha=al, M=M, c=i.c, ct=i.c_tilde, eps=i.eps, Q=i.quad_nodes)
    ref = O.evaluate(pb, O.grid(pb), x, O.OUT_GD)
    assert (np.abs(got - ref) / np.maximum(np.abs(ref), 1e-6 * np.abs(ref).max())).max() < 1e-10
