"""The split gathers' fixed-point stencil and phase against the double plans: positions around the range where
the double form takes over (2^19 grid cells or wave lengths), far beyond it, at stencil nodes and
cell edges, near grid and far-region grid, one and seven fields."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1801_05977_gb300 import gf

pytestmark = pytest.mark.gpu

M = (16, 32, 16)
EDGE = 2.0 ** 19 * 2 * np.pi / 32  # 2^19 cells of the x2 axis


def cloud(far):
    rng = np.random.default_rng(11)
    x = rng.uniform(-1.0, 1.0, (3000, 3))
    x[:1000, :2] *= 20.0
    x[1000:2000, :2] = EDGE * rng.choice([-1.0, 1.0], (1000, 2)) * (1.0 + 2e-2 * x[1000:2000, :2])
    x[2000:, :2] *= 40.0 * EDGE
    x[:300, 0] = rng.integers(-40, 41, 300) * (2 * np.pi / M[0])
    x[:300, 1] = rng.integers(-80, 81, 300) * (2 * np.pi / M[1])
    x[:, 2] *= 0.6
    if far:
        x[:, 2] = np.sign(x[:, 2]) * (0.6 + 1e-9 + np.abs(x[:, 2]) * 0.6)
    t = x[:, :2] - 2 * np.pi * np.rint(x[:, :2] / (2 * np.pi))
    x[np.hypot(np.hypot(t[:, 0], t[:, 1]), x[:, 2]) < 0.05, 2] = 0.3 if not far else 0.8
    return torch.from_numpy(x).cuda()


# float grid, stencil and phase against the double ones: a few 2^-24 of the largest value; the singular part
# and the grid are those of the other comparisons of the two precisions (5e-6 of the largest value)
@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("kind", [gf.GF_HELMHOLTZ, gf.GF_MAXWELL])
def test_fixed_point_positions(kind, far):
    x = cloud(far)
    which = gf.GF_OUT_MAXWELL7 if kind == gf.GF_MAXWELL else gf.GF_OUT_GD
    kw = dict(kind=kind, **(dict(far_grid_M=32) if far else {}))
    out = []
    for precision in (gf.GF_FP64, gf.GF_FP32_SPLIT):
        p = gf.Plan(3, 2.5, (0.1, 0.3), M, precision=precision, **kw)
        out.append(p.eval_points(x, which).cpu().numpy())
        p.close()
    for rows in (slice(0, 1000), slice(1000, 2000), slice(2000, None)):
        err = np.abs(out[1][rows] - out[0][rows]).max(axis=0) / np.abs(out[0]).max(axis=0)
        assert err.max() < 5e-6, (rows, err)
