"""The far series by matrix products (long target lists) against the series kernels (the same
targets in short calls), over what the product path accepts: both precisions, Helmholtz and
Maxwell, few and many propagating indices, clouds that its cells cannot take (left to the
series kernels), one |x3| for all targets, lattice cells away from the first, ragged tails."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf
from paper_1801_05977_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# the products keep 2^-60 (split: 2^-30) of the largest term of each target's series per
# weight and phase, the series kernels their working precision; both sum about 1e4 terms
TOL = {gf.GF_FP64: 1e-12, gf.GF_FP32_SPLIT: 5e-6}


def cloud(kind, n, seed):
    x = W.targets_3d(n, seed=seed)
    rng = np.random.default_rng(seed)
    sgn = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    if kind == "slab":            # every target far, in a narrow range next to the slab
        x[:, 2] = sgn * rng.uniform(0.6 + 1e-12, 0.62, n)
    elif kind == "one":           # a single |x3|
        x[:, 2] = sgn * 0.75
    elif kind == "wide":          # up to many wavelengths: cells too wide for the expansion
        x[:, 2] = sgn * np.exp(rng.uniform(np.log(0.6), np.log(40.0), n))
    elif kind == "cells":         # other lattice cells, and phases at multiples of a quarter turn
        x[:, :2] += 2 * np.pi * rng.integers(-9, 10, (n, 2))
        x[:64, 0] = np.pi / 2 * rng.integers(-8, 8, 64)
        x[:64, 1] = np.pi / 2 * rng.integers(-8, 8, 64)
        x[:64, 2] = 0.7
    return x


def both(plan, x, which, chunk=4096):
    xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    a = plan.eval_points(xd, which)
    assert torch.equal(a.view(torch.float32 if a.dtype == torch.complex64 else torch.float64),
                       plan.eval_points(xd, which).view(torch.float32 if a.dtype == torch.complex64 else torch.float64))
    b = torch.cat([plan.eval_points(xd[i:i + chunk], which) for i in range(0, x.shape[0], chunk)])
    return a.cpu().numpy().astype(np.complex128), b.cpu().numpy().astype(np.complex128)


def check(plan, x, which, tol):
    a, b = both(plan, x, which)
    far = np.abs(x[:, 2]) > 0.6
    assert np.isfinite(a).all()
    e = np.abs(a - b)[far].max(axis=0) / np.abs(b[far]).max(axis=0)
    assert e.max() < tol, e
    assert np.array_equal(a[~far], b[~far])
    assert plan.status() == gf.GF_OK


@pytest.mark.parametrize("k,alpha", [(0.4, (0.1, 0.3)), (0.5, (0.3, 0.3)), (0.2, (0.4, -0.4)), (2.5, (0.1, 0.3)), (4.9, (-0.47, 0.08)), (6.8, (0.0, 0.25)), (7.3, (0.2, 0.1))])
@pytest.mark.parametrize("kind", ["uniform", "slab", "wide"])
def test_helmholtz_fp64(k, alpha, kind):
    plan = gf.Plan(3, k, alpha, (32, 32, 16))
    check(plan, cloud(kind, 30011, 3), gf.GF_OUT_GD, TOL[gf.GF_FP64])


@pytest.mark.parametrize("n", [12288, 12289, 40000])
@pytest.mark.parametrize("kind", ["one", "cells"])
def test_helmholtz_fp64_tails(n, kind):
    plan = gf.Plan(3, 2.5, (0.1, 0.3), (32, 32, 16))
    check(plan, cloud(kind, n, 5), gf.GF_OUT_GD, TOL[gf.GF_FP64])


@pytest.mark.parametrize("which", [gf.GF_OUT_MAXWELL6, gf.GF_OUT_MAXWELL7])
@pytest.mark.parametrize("k,kind", [(2.5, "uniform"), (1.1, "slab"), (4.2, "cells"), (2.5, "wide")])
def test_maxwell_fp64(which, k, kind):
    plan = gf.Plan(3, k, (0.1, 0.3), (32, 32, 16), kind=gf.GF_MAXWELL)
    # the series kernels' float tails bound this comparison (up to 1e-11 of an entry's maximum)
    check(plan, cloud(kind, 40003, 7), which, 5e-11)


@pytest.mark.parametrize("k,kind", [(0.4, "uniform"), (2.5, "slab"), (4.9, "wide"), (2.5, "cells")])
def test_helmholtz_split(k, kind):
    plan = gf.Plan(3, k, (0.1, 0.3), (32, 32, 16), precision=gf.GF_FP32_SPLIT)
    check(plan, cloud(kind, 200003, 9), gf.GF_OUT_GD, TOL[gf.GF_FP32_SPLIT])


@pytest.mark.parametrize("k,kind", [(2.5, "uniform"), (4.2, "slab")])
def test_maxwell_split(k, kind):
    plan = gf.Plan(3, k, (0.1, 0.3), (32, 32, 16), precision=gf.GF_FP32_SPLIT, kind=gf.GF_MAXWELL)
    check(plan, cloud(kind, 330001, 11), gf.GF_OUT_MAXWELL7, TOL[gf.GF_FP32_SPLIT])


def test_long_list_with_far_grid_keeps_the_series_beyond_it():
    """A plan with a far-region grid keeps its own route (|x3| > zmax by the series kernels)."""
    plan = gf.Plan(3, 2.5, (0.1, 0.3), (32, 32, 16), precision=gf.GF_FP32_SPLIT, far_grid_M=64)
    x = cloud("wide", 200003, 13)
    a, b = both(plan, x, gf.GF_OUT_GD)
    assert np.abs(a - b).max() < 1e-6 * np.abs(b).max()
