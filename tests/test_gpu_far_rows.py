"""Far lists whose targets have few rows of the series (large c): row slabs of two rows and more, lists of one chunk,
short and long ones, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,ct", [(1.2, 1.6), (3.0, 4.0), (12.0, 16.0)])
@pytest.mark.parametrize("n", [5, 700, 5000, 12000])
def test_far_rows(c, ct, n):
    rng = np.random.default_rng(n)
    x = np.c_[rng.uniform(-7.0, 7.0, (n, 2)), rng.uniform(c + 1e-9, ct, n) * rng.choice([-1.0, 1.0], n)]
    ref = slice(0, n, max(1, n // 200))
    plan = gf.Plan(3, 2.5, (0.1, 0.3), (16, 16, 16), c=c, c_tilde=ct)
    got = plan.eval_points(torch.from_numpy(x).cuda(), gf.GF_OUT_GD).cpu().numpy()[ref]
    i = plan.info
    pb = O.Problem(dim=3, k=2.5, alpha=(0.1, 0.3), M=(16, 16, 16), c=i.c, ct=i.c_tilde, eps=i.eps, Q=i.quad_nodes)
    plan.close()
    want = O.evaluate(pb, O.grid(pb), x[ref], O.OUT_GD)
    # normwise, as the other double-precision comparisons with the oracle
    assert np.abs(got - want).max() < 1e-12 * np.abs(want).max()
