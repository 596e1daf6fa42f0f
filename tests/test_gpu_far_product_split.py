"""The split plans' Helmholtz products (lists from 786432 targets on) against the series kernels (the same targets in
short calls): none, few and many propagating indices, clouds whose cells the products take, partly take and leave
(one and two targets a lane in the series kernel, a ragged last cell among them), lattice cells away from the first.
That the products ran is seen by their three launches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu

# as the products' other split tests: 2^-30 of the largest term per weight and phase against float sums of 3000 terms
TOL = 5e-6


def cloud(kind, n, seed):
    rng = np.random.default_rng(seed)
    x = np.empty((n, 3))
    x[:, :2] = rng.uniform(0.0, 2.0 * np.pi, (n, 2))
    z = rng.uniform(-1.0, 1.0, n)
    sgn = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    if kind == "slab":
        z = sgn * rng.uniform(0.6 + 1e-12, 0.62, n)
    elif kind == "wide":          # cells too wide in |x3|, from the second on
        z = sgn * np.exp(rng.uniform(np.log(0.6), np.log(40.0), n))
    elif kind == "mixed":         # a narrow slab, then a thin tail: cells taken, then cells left over
        z = sgn * np.where(rng.random(n) < 0.9, rng.uniform(0.6 + 1e-12, 0.7, n), rng.uniform(2.0, 9.0, n))
    elif kind == "cells":
        x[:, :2] += 2 * np.pi * rng.integers(-9, 10, (n, 2))
        x[:64, :2] = np.pi / 2 * rng.integers(-8, 8, (64, 2))
        z[:64] = 0.7
    x[:, 2] = z
    return torch.from_numpy(x).cuda()


@pytest.mark.parametrize("n", [786433, 800003])
@pytest.mark.parametrize("k,kind", [(0.4, "uniform"), (2.5, "slab"), (4.9, "wide"), (2.5, "mixed"), (0.4, "mixed"), (2.5, "cells"), (6.8, "uniform")])
def test_split(k, kind, n):
    plan = gf.Plan(3, k, (0.1, 0.3), (32, 32, 16), precision=gf.GF_FP32_SPLIT)
    x = cloud(kind, n, 9)
    short = gf.launch_count()
    plan.eval_points(x[:1000], gf.GF_OUT_GD)
    short = gf.launch_count() - short
    long = gf.launch_count()
    a = plan.eval_points(x, gf.GF_OUT_GD)
    long = gf.launch_count() - long
    assert long == short + 3
    b = torch.cat([plan.eval_points(v, gf.GF_OUT_GD) for v in x.split(65536)])
    far = x[:, 2].abs() > 0.6
    assert torch.isfinite(torch.view_as_real(a)).all()
    assert torch.equal(torch.view_as_real(a[~far]), torch.view_as_real(b[~far]))
    assert float((a - b)[far].abs().max() / b[far].abs().max()) < TOL
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(plan.eval_points(x, gf.GF_OUT_GD)))
    assert plan.status() == gf.GF_OK
    plan.close()
