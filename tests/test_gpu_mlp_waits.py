"""The training pass after a bounded wait that ran out in one warp only: every warp of the CTA
has to leave, whichever product the warp gave up at (before, at and after the head's barriers, in a CTA's
first tile and in its second), the error word says so, and the network goes on as before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


def samples(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    return torch.rand(n, 6, generator=g, device="cuda"), torch.randn(n, 2, generator=g, device="cuda")


@pytest.mark.parametrize("n,warp,step", [(300, 5, 3), (300, 0, 0), (300, 15, 2), (300, 9, 5), (20000, 3, 6), (20000, 12, 10)])
def test_one_warp_gives_up(n, warp, step):
    mlp = gf.MLP(seed=2)
    x, t = samples(n)
    g, loss = mlp.gradients(x, t)
    assert mlp.wait_selftest(x, t, -1, 0) == gf.GF_OK
    assert mlp.wait_selftest(x, t, warp, step) == gf.GF_ERR_TIMEOUT
    assert mlp.error_word() == 0
    g2, loss2 = mlp.gradients(x, t)
    assert np.array_equal(g, g2) and loss == loss2
    mlp.close()
