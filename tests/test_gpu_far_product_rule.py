"""Which evaluations take the matrix products (three more launches), by the number of targets and c, on both sides of
the line, and the same values as in short calls on either route."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu


def launches(plan, x, which):
    n0 = gf.launch_count()
    out = plan.eval_points(x, which)
    return gf.launch_count() - n0, out


@pytest.mark.parametrize("kind,which,c,ct,n,products", [
    (gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 0.6, 1.0, 12287, False), (gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 0.6, 1.0, 12288, True),
    (gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 0.3, 1.0, 12288, True), (gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 1.2, 1.6, 32000, False),
    (gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 1.2, 1.6, 33000, True), (gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 3.0, 4.0, 100003, False),
    (gf.GF_HELMHOLTZ, gf.GF_OUT_GD, 3.0, 4.0, 200001, True), (gf.GF_MAXWELL, gf.GF_OUT_MAXWELL6, 1.2, 1.6, 40001, False),
    (gf.GF_MAXWELL, gf.GF_OUT_MAXWELL6, 1.2, 1.6, 60001, True)])
def test_route(kind, which, c, ct, n, products):
    plan = gf.Plan(3, 2.5, (0.1, 0.3), (16, 16, 32), kind=kind, c=c, c_tilde=ct)
    rng = np.random.default_rng(n)
    x = torch.from_numpy(np.c_[rng.uniform(-7.0, 7.0, (n, 2)), rng.uniform(c + 1e-9, ct, n) * rng.choice([-1.0, 1.0], n)]).cuda()
    short, _ = launches(plan, x[:1000], which)
    got, out = launches(plan, x, which)
    assert got - short == (3 if products else 0)
    ref = torch.cat([plan.eval_points(v, which) for v in x.split(10000)])
    # the series kernels' float tails bound the Maxwell comparison (as in the products' own test)
    e = (out - ref).abs().amax(0) / ref.abs().amax(0)
    assert float(e.max()) < (1e-12 if kind == gf.GF_HELMHOLTZ else 5e-11)
    plan.close()
