"""The near branch by warps (listed targets) against one thread a target (the allocation-free
evaluation) and, in double, against the oracle: list lengths around a warp, every target next to a source (the
queue of singular parts overflows at once) or none, stencil nodes and cell edges, both signs of
x3 and the slab's faces, distant lattice cells, the remainder alone, the far-region grid."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu

M = (16, 32, 16)
# a few roundings of the stencil's and the singular part's largest term
TOL = {gf.GF_FP64: 1e-12, gf.GF_FP32_SPLIT: 2e-6}


def cloud(kind, n):
    rng = np.random.default_rng(n)
    x = np.empty((n, 3))
    if kind == "source":
        x[:] = rng.normal(size=(n, 3)) * 0.2
        x[:, 2] = np.clip(x[:, 2], -0.6, 0.6)
        x[:, :2] += 2 * np.pi * rng.integers(-2, 3, (n, 2))
    elif kind == "edges":
        x[:, 0] = rng.integers(-16, 17, n) * (2 * np.pi / M[0])
        x[:, 1] = rng.integers(-32, 33, n) * (2 * np.pi / M[1])
        x[:, 2] = rng.choice([-0.6, -0.5, -0.125, 0.0, 0.125, 0.375, 0.6], n)
        x[np.hypot(*(x[:, :2] - 2 * np.pi * np.rint(x[:, :2] / (2 * np.pi))).T) < 1e-9, 2] = 0.3
    elif kind == "cells":
        x[:, :2] = rng.uniform(-3e3, 3e3, (n, 2))
        x[:, 2] = rng.uniform(-0.6, 0.6, n)
    else:  # away from the sources
        x[:, :2] = rng.uniform(1.2, 5.0, (n, 2))
        x[:, 2] = rng.uniform(-0.6, 0.6, n)
    return x


def both(plan, x, which):
    xd = torch.from_numpy(x).cuda()
    a = plan.eval_points(xd, which)
    b = torch.empty_like(a)
    plan.eval_points_noalloc_into(xd, b, which)
    return a.cpu().numpy(), b.cpu().numpy()


@pytest.mark.parametrize("precision", [gf.GF_FP64, gf.GF_FP32_SPLIT])
@pytest.mark.parametrize("kind", [gf.GF_HELMHOLTZ, gf.GF_MAXWELL])
@pytest.mark.parametrize("name,n", [("source", 1), ("source", 700), ("edges", 33), ("edges", 800), ("cells", 31),
                                    ("cells", 2000), ("clear", 32), ("clear", 129)])
def test_list_against_single_threads(name, n, kind, precision):
    x = cloud(name, n)
    outs = [gf.GF_OUT_MAXWELL6, gf.GF_OUT_MAXWELL7] if kind == gf.GF_MAXWELL else [gf.GF_OUT_GD, gf.GF_OUT_LD]
    p = gf.Plan(3, 2.5, (0.1, 0.3), M, precision=precision, kind=kind)
    for which in outs:
        a, b = both(p, x, which)
        assert np.isfinite(a.view(a.real.dtype)).all()
        # per target and entry, against the target's largest entry or the entry's typical size
        scale = np.maximum(np.abs(b).max(axis=1, keepdims=True), np.median(np.abs(b), axis=0))
        assert (np.abs(a - b) / scale).max() < TOL[precision], which
    if precision == gf.GF_FP64 and kind == gf.GF_HELMHOLTZ:
        pb = O.Problem(dim=3, k=2.5, alpha=(0.1, 0.3), M=M)
        ref = O.evaluate(pb, O.grid(pb), x, O.OUT_GD)
        a = both(p, x, gf.GF_OUT_GD)[0]
        # x reduced to its cell keeps a rounding of x: 3e3 ulps of 1 for the distant cells, times k and the
        # gradient next to a source
        assert (np.abs(a - ref) / np.abs(ref)).max() < (1e-9 if name == "cells" else 1e-10)
    p.close()


@pytest.mark.parametrize("precision", [gf.GF_FP64, gf.GF_FP32_SPLIT])
@pytest.mark.parametrize("kind", [gf.GF_HELMHOLTZ, gf.GF_MAXWELL])
def test_far_grid_list(kind, precision):
    x = cloud("cells", 1500)
    rng = np.random.default_rng(1)
    x[:, 2] = rng.choice([-1.0, 1.0], len(x)) * rng.uniform(0.6, 1.0, len(x))
    x[:6, 2] = (0.6, np.nextafter(0.6, 1), -np.nextafter(0.6, 1), 1.0, -1.0, np.nextafter(1.0, 0))
    p = gf.Plan(3, 2.5, (0.1, 0.3), M, precision=precision, kind=kind, far_grid_M=32)
    a, b = both(p, x, gf.GF_OUT_MAXWELL7 if kind == gf.GF_MAXWELL else gf.GF_OUT_GD)
    assert (np.abs(a - b).max(axis=0) / np.abs(b).max(axis=0)).max() < TOL[precision]
    p.close()
