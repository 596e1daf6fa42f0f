"""The far series' matrix products after a bounded wait that ran out in one warp: copies, MMAs or sums,
at the first hand-over, in the middle and beyond one tile.  Every warp of the CTA has to leave with its copies
landed and its MMAs done, the status says so, and the plan evaluates as before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf
from paper_1801_05977_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# far tiles beyond one per CTA (152 CTAs: 40% of the targets over 128 x 152)
@pytest.mark.parametrize("precision,kind,which,n", [(gf.GF_FP64, gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 100003),
                                                    (gf.GF_FP32_SPLIT, gf.GF_MAXWELL, gf.GF_OUT_MAXWELL6, 330001)])
@pytest.mark.parametrize("warp,unit", [(0, 0), (0, 3), (1, 0), (2, 5), (3, 30), (4, 0), (4, 2)])
def test_one_warp_gives_up(precision, kind, which, n, warp, unit):
    plan = gf.Plan(3, 2.5, (0.1, 0.3), (16, 16, 16), precision=precision, kind=kind)
    x = torch.from_numpy(W.targets_3d(n, seed=3)).cuda()
    a = plan.eval_points(x, which)
    out = torch.empty_like(a)
    assert plan.wait_selftest(x, out, which, 1, -1) == gf.GF_OK
    assert torch.equal(torch.view_as_real(out), torch.view_as_real(a))
    assert plan.wait_selftest(x, out, which, warp, unit) == gf.GF_ERR_TIMEOUT
    assert plan.status() == gf.GF_OK
    assert torch.equal(torch.view_as_real(plan.eval_points(x, which)), torch.view_as_real(a))
    plan.close()
