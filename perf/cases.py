"""Performance cases: the calls that users of this framework make, at the sizes they make them.

`listed()` gives the fixed cases and `draw(rng)` further ones of the same ranges; `prepare` makes what a
program has in hand before the call (targets, and the plan, batch or network where a program keeps one),
`run` is one pass through the public entry points, `work` the bytes and operations a pass cannot do
without, and `exact` the same outputs in 64 bits from plain torch, without the library's code.

Kinds of case (`kind`):
  gd       3D doubly quasi-periodic G_d: `call` "step" builds the plan, evaluates and releases it (a solver
           that moves through wave numbers), "eval" evaluates with a plan in hand (a solver's inner loop),
           "host" does so with host buffers in and out
  maxwell  the Maxwell Green's tensor (six entries, or seven with G_d), the same calls
  g2d      2D quasi-periodic G: plan and evaluation
  deriv2d  2D first derivatives and differences of second derivatives: plan and both outputs
  sweep    a batched (alpha, k) sweep as one graph: synthesis and evaluation of every pair
  forward  the surrogate network's fused forward pass
  train    optimizer steps of the surrogate network, then a copy of its parameters (a checkpoint)
"""
import math

import numpy as np
import torch

from paper_1801_05977_gb300 import gf

PI, TWO_PI = math.pi, 2.0 * math.pi


def listed():
    return [
        # the headline step: one wave number, double precision, a million targets
        dict(name="gd_fp64_step_1e6", kind="gd", call="step", prec="fp64", k=2.5, a1=0.1, a2=0.3, m=128, m3=64, n=1000000),
        # a small call with the plan in hand: latency and launches
        dict(name="gd_fp64_eval_1017", kind="gd", call="eval", prec="fp64", k=2.5, a1=0.1, a2=0.3, m=64, m3=32, n=1017),
        # an ordinary call from host memory, pinned buffers, plan in hand
        dict(name="gd_fp64_host_1e5", kind="gd", call="host", prec="fp64", k=3.7, a1=-0.2, a2=0.45, m=128, m3=64, n=100003),
        # the same step in split precision, and with the far-region grid
        dict(name="gd_split_step_1e6", kind="gd", call="step", prec="split", k=2.5, a1=0.1, a2=0.3, m=128, m3=64, n=1000000),
        dict(name="gd_split_fargrid_1e6", kind="gd", call="step", prec="split", k=2.5, a1=0.1, a2=0.3, m=128, m3=64,
             far=512, n=1000000),
        # Maxwell tensor: the large clustered cloud in split precision; seven entries in double precision
        dict(name="maxwell_split_step_1e6", kind="maxwell", call="step", prec="split", k=2.5, a1=0.1, a2=0.3, m=256, m3=64,
             entries=6, n=1000000),
        dict(name="maxwell_fp64_eval_1e5", kind="maxwell", call="eval", prec="fp64", k=2.5, a1=0.1, a2=0.3, m=64, m3=32,
             entries=7, n=100003),
        # 2D: the small classic configuration, and the derivatives on a fine grid
        dict(name="g2d_fp64_step_1e4", kind="g2d", prec="fp64", k=1.3, a1=0.2, m=64, n=10000),
        dict(name="deriv2d_fp64_step_1e5", kind="deriv2d", prec="fp64", k=1.3, k2=2.1, a1=0.2, m=256, n=100000),
        # a Bloch / frequency sweep: 64 pairs with their own grids, ragged target counts
        dict(name="sweep_split_64x1e5", kind="sweep", prec="split", pairs=64, per=100000),
        # the surrogate network: inference, and a stretch of training
        dict(name="mlp_forward_3e5", kind="forward", n=300001),
        dict(name="mlp_train_4x8192", kind="train", n=8192, steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pair(rng, kmin, kmax):
    """(k, alpha1, alpha2) clear of Wood anomalies by 1e-2."""
    while True:
        k, a1, a2 = rng.uniform(kmin, kmax), rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5)
        if min(abs(math.hypot(a1 + i, a2 + j) - k) for i in range(-7, 8) for j in range(-7, 8)) > 1e-2:
            return round(k, 6), round(a1, 6), round(a2, 6)


def draw(rng):
    kind = rng.choice(["gd", "gd", "gd", "gd", "maxwell", "maxwell", "g2d", "deriv2d", "sweep", "forward", "train"])
    k, a1, a2 = _pair(rng, 0.5, 5.0)
    prec = rng.choice(["fp64", "split"])
    m = min(256, max(32, 2 ** math.ceil(math.log2(math.ceil(32 * k)))))
    if kind == "gd":
        c = dict(kind=kind, call=rng.choice(["step", "eval", "host"]), prec=prec, k=k, a1=a1, a2=a2, m=min(m, 128), m3=rng.choice([32, 64]),
                 n=_log_int(rng, 500, 1000000))
        if prec == "split" and rng.random() < 0.3:
            c["far"] = rng.choice([128, 256, 512])
        return c
    if kind == "maxwell":
        return dict(kind=kind, call=rng.choice(["step", "eval"]), prec=prec, k=k, a1=a1, a2=a2, m=min(m, 128), m3=rng.choice([32, 64]),
                    entries=rng.choice([6, 7]), n=_log_int(rng, 500, 1000000 if prec == "split" else 100000))
    if kind in ("g2d", "deriv2d"):
        k2 = {} if kind == "g2d" else {"k2": round(k + rng.uniform(0.3, 1.5), 6)}
        while min(abs(abs(a1 + i) - v) for i in range(-8, 9) for v in [k, *k2.values()]) < 1e-2:
            a1 = round(rng.uniform(-0.5, 0.5), 6)
        return dict(kind=kind, prec=prec, k=k, a1=a1, m=rng.choice([64, 128, 256]), n=_log_int(rng, 500, 100000), **k2)
    if kind == "sweep":
        return dict(kind=kind, prec="split", pairs=rng.randint(8, 64), per=_log_int(rng, 2000, 100000))
    if kind == "forward":
        return dict(kind=kind, n=_log_int(rng, 1000, 1000000))
    return dict(kind=kind, n=_log_int(rng, 1024, 16384), steps=rng.randint(1, 4))


# --------------------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _cloud3(n, g, clustered=False):
    """x1, x2 ~ U[0, 2 pi), x3 ~ U[-1, 1], none within 1e-3 of a lattice point; clustered: a tenth of them in
    the shell 1e-3 <= r <= 0.05 around the cell's corners (where the singular part dominates)."""
    x = torch.stack([_uniform(g, n, 0.0, TWO_PI), _uniform(g, n, 0.0, TWO_PI), _uniform(g, n, -1.0, 1.0)], 1)
    if clustered:
        r = (1e-9 + torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (0.05 ** 3 - 1e-9)) ** (1.0 / 3.0)
        d = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
        y = d / d.norm(dim=1, keepdim=True) * r[:, None]
        y[:, :2] += TWO_PI * torch.randint(0, 2, (n, 2), generator=g, device="cuda").double()
        x = torch.where((torch.rand(n, generator=g, device="cuda") < 0.1)[:, None], y, x)
    d = x[:, :2] - TWO_PI * torch.round(x[:, :2] / TWO_PI)
    near = (d.square().sum(1) + x[:, 2].square()).sqrt() < 1e-3
    x[:, 2] = torch.where(near, torch.full_like(x[:, 2], 0.05), x[:, 2])
    return x.contiguous()


def _cloud2(n, g):
    x = torch.stack([_uniform(g, n, 0.0, TWO_PI), _uniform(g, n, -1.0, 1.0)], 1)
    d = x[:, 0] - TWO_PI * torch.round(x[:, 0] / TWO_PI)
    near = (d.square() + x[:, 1].square()).sqrt() < 1e-3
    x[:, 1] = torch.where(near, torch.full_like(x[:, 1], 0.05), x[:, 1])
    return x.contiguous()


def _points(case, seed):
    g = _gen(seed)
    if case["kind"] == "gd":
        return _cloud3(case["n"], g)
    if case["kind"] == "maxwell":
        return _cloud3(case["n"], g, clustered=True)
    return _cloud2(case["n"], g)


def _prec(case):
    return gf.GF_FP64 if case["prec"] == "fp64" else gf.GF_FP32_SPLIT


def _which(case):
    return {"gd": gf.GF_OUT_GD, "g2d": gf.GF_OUT_G}.get(case["kind"]) if case["kind"] != "maxwell" else (
        gf.GF_OUT_MAXWELL6 if case["entries"] == 6 else gf.GF_OUT_MAXWELL7)


def _plan(case):
    p = _prec(case)
    if case["kind"] == "gd":
        return gf.Plan(3, case["k"], (case["a1"], case["a2"]), (case["m"], case["m"], case["m3"]), precision=p,
                       far_grid_M=case.get("far", 0))
    if case["kind"] == "maxwell":
        return gf.Plan(3, case["k"], (case["a1"], case["a2"]), (case["m"], case["m"], case["m3"]), precision=p, kind=gf.GF_MAXWELL)
    if case["kind"] == "g2d":
        return gf.Plan(2, case["k"], (case["a1"],), (case["m"], case["m"]), precision=p)
    return gf.Plan(2, case["k"], (case["a1"],), (case["m"], case["m"]), precision=p, kind=gf.GF_DERIV2D, k2=case["k2"], c_tilde=1.4)


def _sweep_sizes(case):
    """The sweep's pairs (fixed by their number), grids (32 points per wave number, 32 to 256) and ragged
    target counts."""
    rng = np.random.Generator(np.random.PCG64(case["pairs"]))
    k, al = [], []
    while len(k) < case["pairs"]:
        kk, a = rng.uniform(0.5, 5.0), rng.uniform(-0.5, 0.5, 2)
        n = np.arange(-7, 8)
        if np.abs(np.hypot((a[0] + n)[:, None], (a[1] + n)[None, :]) - kk).min() > 1e-3:
            k.append(kk)
            al.append(a)
    k = np.array(k)
    m = np.clip(2 ** np.ceil(np.log2(np.ceil(32 * k))), 32, 256).astype(np.int32)
    M = np.stack([m, m, np.full(len(m), 64, np.int32)], 1)
    per = rng.integers(case["per"] * 3 // 4, case["per"] + 1, case["pairs"])
    return k, np.array(al), M, np.concatenate([[0], np.cumsum(per)]).astype(np.int64)


_MLP_DIMS = [80, 256, 256, 256, 256, 2]


def _mlp_params(seed):
    rng = np.random.default_rng(seed)
    out = []
    for i, o in zip(_MLP_DIMS[:-1], _MLP_DIMS[1:]):
        out += [rng.uniform(-1, 1, o * i) / math.sqrt(i), rng.uniform(-0.05, 0.05, o)]
    return np.concatenate(out).astype(np.float32)


def _mlp_samples(n, seed):
    g = _gen(seed)
    lo = torch.tensor([-PI, -PI, -0.6, -0.5, -0.5, 1.0], device="cuda")
    hi = torch.tensor([PI, PI, 0.6, 0.5, 0.5, 4.0], device="cuda")
    x = lo + (hi - lo) * torch.rand(n, 6, generator=g, device="cuda")
    t = torch.stack([torch.cos(x[:, 0] + x[:, 3] * 2) * torch.exp(-x[:, 2].abs()), torch.sin(x[:, 1] - x[:, 5])], 1)
    return x.contiguous(), (t + 0.05 * torch.randn(n, 2, generator=g, device="cuda")).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "forward":
        net = gf.MLP(seed=1)
        net.set_params(_mlp_params(seed))
        return dict(case=case, net=net, x=_mlp_samples(case["n"], seed)[0])
    if kind == "train":
        net = gf.MLP(seed=1)
        net.set_params(_mlp_params(seed))
        x, t = _mlp_samples(case["n"] * case["steps"], seed)
        return dict(case=case, net=net, x=x, t=t, loss=torch.zeros(case["steps"], dtype=torch.float32, device="cuda"))
    if kind == "sweep":
        k, al, M, off = _sweep_sizes(case)
        batch = gf.Batch(k, al, M, precision=_prec(case))
        n = int(off[-1])
        return dict(case=case, batch=batch, x=_cloud3(n, _gen(seed)), off=off, stream=torch.cuda.Stream(),
                    out=torch.empty((n, 1), dtype=batch.complex_dtype, device="cuda"))
    s = dict(case=case, x=_points(case, seed))
    if case.get("call", "step") != "step":
        s["plan"] = _plan(case)
    if case.get("call") == "host":
        s["x"] = s["x"].cpu().pin_memory()
        s["out"] = torch.empty((case["n"], 1), dtype=s["plan"].complex_dtype).pin_memory()
    return s


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "forward":
        return state["net"].forward(state["x"])
    if kind == "train":
        net, n, loss = state["net"], case["n"], state["loss"]
        for i in range(case["steps"]):
            net.train_step(state["x"][i * n:(i + 1) * n], state["t"][i * n:(i + 1) * n], 1e-4, loss[i:i + 1])
        return {"loss": loss, "params": net.get_params()}
    if kind == "sweep":
        st = state["stream"]
        st.wait_stream(torch.cuda.current_stream())
        state["batch"].run_graph(state["x"], state["off"], state["out"], gf.GF_OUT_GD, stream=st)
        torch.cuda.current_stream().wait_stream(st)
        return state["out"]
    if case.get("call") == "host":
        return state["plan"].eval_points_host(state["x"], state["out"], _which(case))
    if case.get("call") == "eval":
        return state["plan"].eval_points(state["x"], _which(case))
    plan = _plan(case)
    if kind == "deriv2d":
        out = [plan.eval_points(state["x"], gf.GF_OUT_GRAD), plan.eval_points(state["x"], gf.GF_OUT_HESSDIFF)]
    else:
        out = plan.eval_points(state["x"], _which(case))
    plan.close()
    return out


def work(case):
    """Bytes: targets in, values out, and the interpolation grid once where the pass makes it.  Operations: the
    inverse FFTs of the grid, a cubic stencil per near target and the eigenseries' terms per far one."""
    kind = case["kind"]
    if kind in ("forward", "train"):
        w = sum(i * o for i, o in zip(_MLP_DIMS[:-1], _MLP_DIMS[1:]))
        if kind == "forward":
            return {"bytes": 32.0 * case["n"] + 4.0 * w, "flops": 2.0 * w * case["n"]}
        return {"bytes": case["steps"] * (32.0 * case["n"] + 28.0 * w), "flops": 6.0 * w * case["n"] * case["steps"]}
    fp64 = case["prec"] == "fp64"
    el = 16 if fp64 else 8
    if kind == "sweep":
        k, al, M, off = _sweep_sizes(case)
        nodes, n, fields, ent, dim, planes = float((M[:, 0] * M[:, 1]).sum()) * 25, int(off[-1]), 1, 1, 3, 25
    elif kind in ("gd", "maxwell"):
        fields = 1 if kind == "gd" else 7
        ent, n, dim = (1 if kind == "gd" else case["entries"]), case["n"], 3
        nodes = float(case["m"]) ** 2 * case["m3"] * 0.4 if case["call"] == "step" else 0.0
    else:
        fields, ent = (1, 1) if kind == "g2d" else (6, 6)
        n, dim, nodes = case["n"], 2, float(case["m"]) ** 2
    far = 0.0 if case.get("far") else 0.4 * n
    T = math.log(1e16 if fp64 else 1e8) + 3.0
    terms = 1.56 * PI * T * T if dim == 3 else 2.0 * T * 1.28  # mean over 0.6 <= z <= 1 of (T/z)^2 pi, 2 T/z
    per = 10.0 if ent == 1 else 40.0
    flops = nodes * fields * 5.0 * 18 + (n - far) * fields * 4.0 * (4 ** dim) + far * terms * per
    if case.get("far"):
        nodes += float(case["far"]) ** 2 * 19
    return {"bytes": n * (8.0 * dim + el * ent) + nodes * fields * el, "flops": flops}


# --------------------------------------------------------------------------- the same in 64 bits, by plain torch
# The method: G = singular part + smooth quasi-periodic remainder; the remainder's Fourier coefficients on
# a uniform grid, an inverse FFT, tensor cubic interpolation at |x_last| <= c; the eigenseries beyond.

C0, EPS = 0.6, 0.45


def _d64(v):
    return torch.as_tensor(v, dtype=torch.float64, device="cuda")


def _smooth(s, order):
    """The order-8 smoothstep on [0, 1] (order 0) and its first two derivatives."""
    t = torch.clamp(s, 0.0, 1.0)
    if order == 1:
        return 218790.0 * (t * (1 - t)) ** 8
    if order == 2:
        return 8 * 218790.0 * (t * (1 - t)) ** 7 * (1 - 2 * t)
    c = [24310.0, -175032.0, 556920.0, -1021020.0, 1178100.0, -875160.0, 408408.0, -109395.0, 12870.0]

    def low(u):
        v = torch.zeros_like(u)
        for a in reversed(c):
            v = v * u + a
        return v * u ** 9

    return torch.where(t <= 0.5, low(t), 1 - low(1 - t))


def _gauss(a, b, q):
    x, w = np.polynomial.legendre.leggauss(q)
    return _d64(0.5 * (a + b) + 0.5 * (b - a) * x), _d64(0.5 * (b - a) * w)


def _c_tilde(ks, al, M, ct0):
    """c~, moved off the resonances beta = q."""
    n = [np.arange(-m // 2, m // 2) for m in M[:-1]]
    A2 = (al[0] + n[0]) ** 2 if len(n) == 1 else ((al[0] + n[0]) ** 2)[:, None] + ((al[1] + n[1]) ** 2)[None, :]
    ct = ct0
    for t in range(101):
        worst = np.inf
        for k in ks:
            a2 = A2[A2 < k * k]
            q = np.arange(M[-1] // 2 + 1) * PI / ct
            if a2.size:
                worst = min(worst, np.abs(k * k - a2[:, None] - (q * q)[None, :]).min() / (k * k))
        if worst >= 1e-6:
            return ct
        ct = ct0 * (1.0 + 1e-3 * (t + 1))
    return ct


def _freq(m):
    return _d64(np.fft.fftfreq(m, 1.0 / m))


def _xprime(k, A2, q, ct, nq):
    """The cutoff's integral terms of the coefficients, [columns, q]."""
    t, w = _gauss(C0, 0.5 * (C0 + ct), nq)
    wid = 0.5 * (ct - C0)
    X1 = -_smooth((t - C0) / wid, 1) / wid * w
    beta = torch.sqrt(torch.complex(k * k - A2, torch.zeros_like(A2)))
    A = X1 * torch.exp(1j * beta[:, None] * t)
    E = torch.exp(1j * t[:, None] * q)
    return (A @ E.conj()) / (2 * beta[:, None] * (q - beta[:, None])) - (A @ E) / (2 * beta[:, None] * (q + beta[:, None]))


def _cubic(f):
    return [-f * (f - 1) * (f - 2) / 6, (f + 1) * (f - 1) * (f - 2) / 2, -(f + 1) * f * (f - 2) / 2, (f + 1) * f * (f - 1) / 6]


def _cell(x):
    m = torch.floor((x + PI) / TWO_PI)
    return x - TWO_PI * m, m


def _gather(grid, axes):
    """Tensor cubic interpolation: grid [f, N_last, .., N_1], axes = [(u, periodic)] from x1 to the last axis,
    u the position in nodes."""
    st = []
    for (u, per), size in zip(axes, reversed(grid.shape[1:])):
        i0 = torch.floor(u)
        if not per:
            i0 = torch.clamp(i0, 1, size - 3)
        w = _cubic(u - i0)
        st.append([(w[d], (i0.long() + d - 1) % size) for d in range(4)])
    flat = grid.reshape(grid.shape[0], -1)
    out = torch.zeros(grid.shape[0], axes[0][0].numel(), dtype=grid.dtype, device="cuda")

    def walk(level, w, at):
        if level < 0:
            out.add_(w * flat[:, at])
            return
        for ww, ii in st[level]:
            walk(level - 1, ww if w is None else w * ww, ii if at is None else at * grid.shape[-1 - level] + ii)

    walk(len(st) - 1, None, None)
    return out


def _tensor_factors(c1, c2, c3, k):
    return [1 - c1 * c1 / k ** 2, 1 - c2 * c2 / k ** 2, 1 - c3 * c3 / k ** 2, -c1 * c2 / k ** 2, -c1 * c3 / k ** 2, -c2 * c3 / k ** 2,
            torch.ones_like(c1 + c2 + c3)]


def _grid3(k, al, M, ct, maxwell, nq):
    j1, j2, q = _freq(M[0]), _freq(M[1]), _freq(M[2]) * PI / ct
    c1, c2 = (al[0] + j1)[None, :].expand(M[1], M[0]).reshape(-1), (al[1] + j2)[:, None].expand(M[1], M[0]).reshape(-1)
    A2 = c1 * c1 + c2 * c2
    s = torch.sqrt(A2[:, None] + q * q)
    r, w = _gauss(EPS, 2 * EPS, nq)
    u = (r - EPS) / EPS
    B = w * torch.exp(1j * k * r) * (2j * k * (-_smooth(u, 1) / EPS) - _smooth(u, 2) / EPS ** 2)
    h = torch.zeros(s.shape, dtype=torch.complex128, device="cuda")
    for rm, bm in zip(r.tolist(), B.tolist()):
        h += bm * torch.sin(s * rm)
    C = (h / s / (s * s - k * k) + _xprime(k, A2, q, ct, nq)) / (8 * PI ** 2 * ct)
    F = [C] if not maxwell else [f * C for f in _tensor_factors(c1[:, None], c2[:, None], q[None, :], k)]
    n = M[0] * M[1] * M[2]
    return torch.stack([torch.fft.ifftn(f.T.reshape(M[2], M[1], M[0])) * n for f in F])


def _phi(k, r, order):
    s = (r - EPS) / EPS
    Y = [1 - _smooth(s, 0), -_smooth(s, 1) / EPS, -_smooth(s, 2) / EPS ** 2]
    g0 = torch.exp(1j * k * r) / (4 * PI * r)
    g1 = g0 * (1j * k - 1 / r)
    g2 = g0 * ((1j * k - 1 / r) ** 2 + 1 / r ** 2)
    return [g0 * Y[0], g1 * Y[0] + g0 * Y[1], g2 * Y[0] + 2 * g1 * Y[1] + g0 * Y[2]][order]


def _series3(k, al, x, maxwell):
    """The eigenseries at far targets, [entries, n]."""
    n = x.shape[0]
    out = torch.zeros(7 if maxwell else 1, n, dtype=torch.complex128, device="cuda")
    if not n:
        return out
    order = torch.argsort(x[:, 2].abs())
    step = 1024
    for i in range(0, n, step):
        at = order[i:i + step]
        z, sg = x[at, 2].abs(), torch.sign(x[at, 2])
        R = math.sqrt(k * k + (40.0 / float(z.min())) ** 2)
        N = int(R) + 2
        j = _d64(np.arange(-N, N + 1))
        c1, c2 = al[0] + j, al[1] + j
        b2 = c1[:, None] ** 2 + c2[None, :] ** 2 - k * k
        b = torch.sqrt(b2.clamp(min=0))
        e1, e2 = torch.exp(1j * x[at, 0][:, None] * c1), torch.exp(1j * x[at, 1][:, None] * c2)
        ev = b2 > 0
        w = torch.where(ev, torch.exp(-b * z[:, None, None]) / torch.where(ev, b, torch.ones_like(b)), torch.zeros_like(b))

        def summed(v, f2):
            a = torch.complex(torch.bmm(v, (e2.real * f2)[:, :, None])[:, :, 0], torch.bmm(v, (e2.imag * f2)[:, :, None])[:, :, 0])
            return a

        one = torch.ones_like(c2)
        A = summed(w, one)
        tot = [-1j * (e1 * A).sum(1)]
        if maxwell:
            Bs, Cs, wb = summed(w, c2), summed(w, c2 * c2), w * b
            D, E, Fs = summed(wb * b, one), summed(wb, one), summed(wb, c2)
            ik2 = 1 / k ** 2
            rows = [A * (1 - c1 * c1 * ik2), A - Cs * ik2, A + D * ik2, -ik2 * c1 * Bs]
            tot = [-1j * (e1 * v).sum(1) for v in rows] + [sg * (e1 * v).sum(1) for v in (-ik2 * c1 * E, -ik2 * Fs)] + tot
        for p, q in (b2 <= 0).nonzero().tolist():
            be = math.sqrt(-float(b2[p, q]))
            t = torch.exp(1j * be * z) / be * e1[:, p] * e2[:, q]
            f = [1.0]
            if maxwell:
                f = _tensor_factors(c1[p] * torch.ones_like(z), c2[q] * torch.ones_like(z), be * sg, k)
            for e in range(len(tot)):
                tot[e] = tot[e] + f[e] * t
        out[:, at] = torch.stack(tot) * (1j / (8 * PI ** 2))
    return out


def _far_planes(k, al, F, x):
    """Split plans with a far-region grid: the series on planes, tensor cubics between them."""
    ct, nz = 1.0, 16
    hz = (ct - C0) / nz
    z = C0 + hz * (_d64(np.arange(nz + 3)) - 1)
    j = _freq(F)
    d = (al[0] + j)[None, :] ** 2 + (al[1] + j)[:, None] ** 2 - k * k
    beta = torch.sqrt(torch.complex(-d, torch.zeros_like(d)))
    grid = torch.stack([torch.fft.ifft2(1j / (8 * PI ** 2) * torch.exp(1j * beta * zz) / beta) * F * F for zz in z.tolist()])[None]
    t1, m1 = _cell(x[:, 0])
    t2, m2 = _cell(x[:, 1])
    v = _gather(grid, [(t1 * F / TWO_PI, True), (t2 * F / TWO_PI, True), ((x[:, 2].abs() - z[0]) / hz, False)])
    return v * torch.exp(1j * (al[0] * x[:, 0] + al[1] * x[:, 1]))


def _exact3(k, al, M, x, maxwell, entries, far_grid=0):
    ct = _c_tilde([k], al, M, 1.0)
    smax = math.sqrt((M[0] / 2 + 2) ** 2 + (M[1] / 2 + 2) ** 2 + (M[2] / 2 * PI / ct) ** 2)
    nq = max(64, int(smax * EPS / 2) + 32)
    out = torch.zeros(7 if maxwell else 1, x.shape[0], dtype=torch.complex128, device="cuda")
    far = x[:, 2].abs() > C0
    if far_grid:
        xf = x[far]
        out[:, far] = _far_planes(k, al, far_grid, xf)
    else:
        out[:, far] = _series3(k, al, x[far], maxwell)
    grid = _grid3(k, al, M, ct, maxwell, nq)
    y = x[~far]
    t1, m1 = _cell(y[:, 0])
    t2, m2 = _cell(y[:, 1])
    L = _gather(grid, [(t1 * M[0] / TWO_PI, True), (t2 * M[1] / TWO_PI, True), (y[:, 2] * M[2] / (2 * ct), True)])
    ph = al[0] * m1 + al[1] * m2
    lat = torch.exp(2j * PI * (ph - torch.round(ph)))
    v = lat * torch.exp(1j * (al[0] * t1 + al[1] * t2)) * L
    r = torch.sqrt(t1 * t1 + t2 * t2 + y[:, 2] ** 2)
    s = r < 2 * EPS
    rs = torch.where(s, r, torch.ones_like(r))
    P0 = _phi(k, rs, 0)
    if maxwell:
        P1, P2, X = _phi(k, rs, 1), _phi(k, rs, 2), [t1 / rs, t2 / rs, y[:, 2] / rs]
        sing = []
        for p, q in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)):
            dl = 1.0 if p == q else 0.0
            sing.append(dl * P0 + (P2 * X[p] * X[q] + P1 / rs * (dl - X[p] * X[q])) / k ** 2)
        sing = torch.stack(sing + [P0])
    else:
        sing = P0[None]
    out[:, ~far] = v + torch.where(s, lat * sing, torch.zeros_like(sing))
    return out[:entries].T.contiguous()


def _bessel(z, orders):
    """J_n(z), n <= 3, by the trapezoidal rule on Bessel's integral (a quarter of the period, by symmetry)."""
    n = 4 * (int(float(z.max()) / 4) + 16)
    t = _d64(np.arange(n // 4 + 1) * (TWO_PI / n))
    w = torch.full_like(t, 4.0 / n)
    w[0] = w[-1] = 2.0 / n
    p = z[:, None] * torch.sin(t)
    c, s = torch.cos(p), torch.sin(p)
    return [(c if o % 2 == 0 else s) @ (w * (torch.cos(o * t) if o % 2 == 0 else torch.sin(o * t))) for o in orders]


def _grid2(k, k2, a1, M, ct, nq):
    """Remainder fields of the 2D plans: L, and with k2 the five derivative fields."""
    j1, q = _freq(M[0])[:, None], (_freq(M[1]) * PI / ct)[None, :]
    c1 = a1 + j1
    A2 = (c1 * c1).reshape(-1)
    D = c1 * c1 + q * q

    def khat(kk):
        return 1 / (D - kk * kk) + _xprime(kk, A2, q[0], ct, nq)

    r, w = _gauss(EPS, 2 * EPS, nq)
    u = (r - EPS) / EPS
    y0, y1, y2 = 1 - _smooth(u, 0), -_smooth(u, 1) / EPS, -_smooth(u, 2) / EPS ** 2
    ph = (2 + torch.log(r)) * y1 / r + y2 * torch.log(r)
    eta = torch.sqrt(j1 * j1 + q * q)
    zero = eta == 0
    e = torch.where(zero, torch.ones_like(eta), eta)
    ue, inv = torch.unique(eta.reshape(-1), return_inverse=True)

    def radial(weights):
        """sum_m a_m J_n(eta r_m) on the grid for each (n, [(r_m, a_m)...])."""
        sums = [torch.zeros_like(ue) for _ in weights]
        for i, (rm, _) in enumerate(weights[0][1]):
            J = _bessel(ue * rm, [o for o, _ in weights])
            for v, j, (_, ra) in zip(sums, J, weights):
                v += ra[i][1] * j
        return [v[inv].reshape(eta.shape) for v in sums]

    pw = w * ph * r
    S0, S1 = radial([(0, list(zip(r.tolist(), pw.tolist()))), (1, list(zip(r.tolist(), (pw * r).tolist())))])
    F10 = -(0.5 * EPS ** 2 * math.log(EPS) - 0.25 * EPS ** 2 + float((w * r * torch.log(r) * y0).sum()))
    F1 = torch.where(zero, torch.full_like(e, F10), (1 + S0) / e ** 2)
    zf = torch.zeros_like(e)
    f2 = torch.where(zero, zf, (-2 * j1 * F1 - j1 / e * S1) / e ** 2)  # F2 = i f2
    K = khat(k)
    F = [K - F1 - a1 * f2]
    if k2:
        f2y = torch.where(zero, zf, (-2 * q * F1 - q / e * S1) / e ** 2)
        cp, sp = torch.where(zero, zf, j1 / e), torch.where(zero, zf, q / e)
        ra, wa = _gauss(0.0, EPS, nq)
        rr, ww = torch.cat([ra, r]), torch.cat([wa, w * y0])
        Q1, R0, R2, T1, T3 = radial([(o, list(zip(rr.tolist(), (ww * rr ** p).tolist()))) for o, p in ((1, 0), (0, 1), (2, 1), (1, 2), (3, 2))])
        c2, s2, c3, s3 = cp * cp - sp * sp, 2 * cp * sp, cp * (4 * cp * cp - 3), sp * (3 - 4 * sp * sp)
        x11, x22, x12 = PI * (R0 - c2 * R2), PI * (R0 + c2 * R2), -PI * s2 * R2
        x111, x112, x122 = 0.5 * PI * (-3 * cp * T1 + c3 * T3), 0.5 * PI * (-sp * T1 + s3 * T3), 0.5 * PI * (-cp * T1 - c3 * T3)
        H1 = -(0.5 * k * k * TWO_PI * f2 - TWO_PI * cp * Q1 - a1 * x11 - 0.5 * a1 ** 2 * x111) / TWO_PI
        H2 = -(0.5 * k * k * TWO_PI * f2y - TWO_PI * sp * Q1 - a1 * x12 - 0.5 * a1 ** 2 * x112) / TWO_PI
        dk, dK = k * k - k2 * k2, K - khat(k2)
        base = -PI * F1 - a1 * PI * f2
        H11 = dk / TWO_PI * (base + 0.5 * x11 + 0.5 * a1 * x111)
        H12 = dk / TWO_PI * (0.5 * x12 + 0.5 * a1 * x112)
        H22 = dk / TWO_PI * (base + 0.5 * x22 + 0.5 * a1 * x122)
        F += [1j * (c1 * K - H1), 1j * (q * K - H2), -c1 * c1 * dK - H11, -c1 * q * dK - H12, -q * q * dK - H22]
    return torch.stack([torch.fft.ifftn(f.T / (4 * PI * ct)) * (M[0] * M[1]) for f in F])


def _exact2(k, k2, a1, M, x, ct0):
    ct = _c_tilde([k] + ([k2] if k2 else []), [a1], M, ct0)
    smax = math.hypot(M[0] / 2 + 1, (M[1] / 2 + 1) * PI / ct)
    grid = _grid2(k, k2, a1, M, ct, max(96, int(smax * EPS / 2) + 48, int(smax * (ct - C0) / 4) + 48))
    out = torch.zeros(6 if k2 else 1, x.shape[0], dtype=torch.complex128, device="cuda")
    far = x[:, 1].abs() > C0
    y = x[~far]
    t, m = _cell(y[:, 0])
    x2 = y[:, 1]
    v = _gather(grid, [(t * M[0] / TWO_PI, True), (x2 * M[1] / (2 * ct), True)])
    r = torch.sqrt(t * t + x2 * x2)
    s = r < 2 * EPS
    Y = torch.where(s, 1 - _smooth((r - EPS) / EPS, 0), torch.zeros_like(r))
    lr, ir2, i2p = torch.log(r), 1 / (r * r), 1 / TWO_PI
    fa = -lr * Y * i2p
    v[0] += torch.complex(fa, -a1 * t * fa)
    if k2:
        kk = k * k
        v[1] += -i2p * Y * torch.complex(-0.5 * kk * t * lr + t * ir2 - 0.5 * a1 ** 2 * t ** 3 * ir2, -a1 * t * t * ir2)
        v[2] += -i2p * Y * torch.complex(-0.5 * kk * x2 * lr + x2 * ir2 - 0.5 * a1 ** 2 * t * t * x2 * ir2, -a1 * t * x2 * ir2)
        d = (kk - k2 * k2) * i2p * Y
        v[3] += d * torch.complex(0.5 * lr + 0.5 * t * t * ir2, -0.5 * a1 * t * lr - 0.5 * a1 * t ** 3 * ir2)
        v[4] += d * torch.complex(0.5 * t * x2 * ir2, -0.5 * a1 * t * t * x2 * ir2)
        v[5] += d * torch.complex(0.5 * lr + 0.5 * x2 * x2 * ir2, -0.5 * a1 * t * lr - 0.5 * a1 * t * x2 * x2 * ir2)
    out[:, ~far] = v * torch.exp(1j * (a1 * t + TWO_PI * (a1 * m - torch.round(a1 * m))))
    y = x[far]
    z, sg = y[:, 1].abs()[:, None], torch.sign(y[:, 1])[:, None]
    c1 = a1 + _d64(np.arange(-90, 91))

    def term(kk):
        be = torch.sqrt(torch.complex(kk * kk - c1 * c1, torch.zeros_like(c1)))
        return be, torch.exp(1j * (be * z + c1 * y[:, 0][:, None]))

    be, E = term(k)
    f = [(E / be).sum(1)]
    if k2:
        be2, E2 = term(k2)
        f += [(1j * c1 * E / be).sum(1), (1j * sg * E).sum(1), (-c1 * c1 * (E / be - E2 / be2)).sum(1), (-c1 * sg * (E - E2)).sum(1),
              (-(be * E - be2 * E2)).sum(1)]
    out[:, far] = torch.stack(f) * (0.25j / PI)
    return out


def _mlp_features(x):
    t1, t2, x3 = x[:, 0], x[:, 1], x[:, 2]
    fr = [(a, b, c) for c in range(2) for a in (-1, 0, 1) for b in (-1, 0, 1) if a or b or c]
    fr += [(0, 0, 2), (0, 0, 3), (2, 0, 0), (-2, 0, 0), (0, 2, 0), (0, -2, 0), (2, 0, 1), (0, 2, 1), (3, 0, 0), (0, 3, 0), (-3, 0, 0),
           (0, -3, 0), (1, 1, 2), (-1, 1, 2), (2, 2, 0)]
    ph = x[:, :3] @ (_d64(fr).T * _d64([1.0, 1.0, PI])[:, None])
    r = torch.sqrt(t1 * t1 + t2 * t2 + x3 * x3)
    return torch.cat([torch.stack([torch.cos(ph), torch.sin(ph)], 2).reshape(x.shape[0], 64), 2 * x[:, 3:5], (x[:, 5:6] - 2.5) / 1.5, r[:, None],
                      torch.exp(-0.5 * ((r[:, None] - 0.15 * _d64(np.arange(12))) / 0.15) ** 2)], 1)


def _mlp_unpack(p):
    out, at = [], 0
    for i, o in zip(_MLP_DIMS[:-1], _MLP_DIMS[1:]):
        out += [p[at:at + o * i].reshape(o, i), p[at + o * i:at + o * i + o]]
        at += o * i + o
    return out


def _mlp(p, x):
    w, h = _mlp_unpack(p), _mlp_features(x)
    for j in range(4):
        h = torch.nn.functional.silu(h @ w[2 * j].T + w[2 * j + 1])
    return h @ w[8].T + w[9]


def exact(case, seed):
    kind = case["kind"]
    if kind == "forward":
        p, x = _d64(_mlp_params(seed)), _mlp_samples(case["n"], seed)[0].double()
        return torch.cat([_mlp(p, x[i:i + 65536]) for i in range(0, x.shape[0], 65536)])
    if kind == "train":
        p = _d64(_mlp_params(seed)).requires_grad_(True)
        x, t = (v.double() for v in _mlp_samples(case["n"] * case["steps"], seed))
        m, v, losses, n = torch.zeros_like(p), torch.zeros_like(p), [], case["n"]
        for i in range(case["steps"]):
            loss = 0.5 * (_mlp(p, x[i * n:(i + 1) * n]) - t[i * n:(i + 1) * n]).square().sum() / n
            (g,) = torch.autograd.grad(loss, p)
            losses.append(loss.detach())
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            step = 1e-4 * (m / (1 - 0.9 ** (i + 1))) / (torch.sqrt(v / (1 - 0.999 ** (i + 1))) + 1e-8)
            p = (p.detach() - step).requires_grad_(True)
        return {"loss": torch.stack(losses), "params": p.detach().cpu().numpy()}
    if kind == "sweep":
        k, al, M, off = _sweep_sizes(case)
        x = _cloud3(int(off[-1]), _gen(seed))
        return torch.cat([_exact3(float(k[i]), [float(v) for v in al[i]], [int(v) for v in M[i]], x[off[i]:off[i + 1]], False, 1)
                          for i in range(len(k))])
    x = _points(case, seed)
    if kind in ("gd", "maxwell"):
        return _exact3(case["k"], [case["a1"], case["a2"]], [case["m"], case["m"], case["m3"]], x, kind == "maxwell",
                       1 if kind == "gd" else case["entries"], case.get("far", 0))
    if kind == "g2d":
        return _exact2(case["k"], 0.0, case["a1"], [case["m"], case["m"]], x, 1.0).T.contiguous()
    v = _exact2(case["k"], case["k2"], case["a1"], [case["m"], case["m"]], x, 1.4)
    return [v[:3].T.contiguous(), v[3:].T.contiguous()]
