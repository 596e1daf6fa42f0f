"""G_d beside the Maxwell entries at small k, where the entries are 1/k^2 times as large: long lists keep it as
close to the oracle as short ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,ulp", [(gf.GF_FP64, 25001, 2.0 ** -53), (gf.GF_FP32_SPLIT, 330001, 2.0 ** -24)])
@pytest.mark.parametrize("k", [0.005, 0.05, 0.21])
def test_gd_entry(precision, n, ulp, k):
    """The series kernels' error is their float tails' (double) or their sums' (split); a long list may add 32
    roundings of the largest value, the sums of about 1e4 terms' worth (their square root, a third of a rounding each)."""
    rng = np.random.default_rng(n)
    x = np.c_[rng.uniform(-7.0, 7.0, (n, 2)), rng.uniform(0.6 + 1e-9, 1.0, n) * rng.choice([-1.0, 1.0], n)]
    xd = torch.from_numpy(x).cuda()
    plan = gf.Plan(3, k, (0.1, 0.3), (16, 16, 16), precision=precision, kind=gf.GF_MAXWELL)
    i = plan.info
    at = np.arange(0, n, n // 400)
    long = plan.eval_points(xd, gf.GF_OUT_MAXWELL7)[:, 6].cpu().numpy()[at]
    short = plan.eval_points(xd[torch.from_numpy(at).cuda()].contiguous(), gf.GF_OUT_MAXWELL7)[:, 6].cpu().numpy()
    plan.close()
    pb = O.Problem(dim=3, k=k, alpha=(0.1, 0.3), M=(16, 16, 16), c=i.c, ct=i.c_tilde, eps=i.eps, Q=i.quad_nodes)
    ref = O.evaluate(pb, O.grid(pb), x[at], O.OUT_GD)[:, 0]
    el, es = (np.abs(v - ref).max() / np.abs(ref).max() for v in (long, short))
    assert el < es + 32 * ulp, (el, es)
