"""Workloads of the immersed-boundary propagator for timing and comparison.

Each case is one call, or one short sequence of calls, that a user of the library
makes: build the modified stencils of a topography, propagate a shot (second order or
staggered, 2D or 3D, FP32 or FP64), propagate or differentiate a batch of shots, take a
training step of the learned-stencil network.  ``prepare`` makes the inputs and whatever
a program keeps between calls (tables, the network), ``run`` makes the calls, ``exact``
restates the result in 64 bits with plain torch (its own boundary points, fits and time
loop; nothing of the library).

Grids are sizes of this repository's configurations, tests and benchmark, or in their
range; h = 10 m (5 m for the staggered form), topographies are seeded sums of Gaussian
hills or sinusoids, velocities 1500-4000 m/s.
"""
import itertools
import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_2309_03600_gb300 import ib, inputs

DEV = "cuda"
CMAX = 4000.0
LAYER = 20                      # absorbing layer (nodes) where a case has one


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The smallest shot: the 201 x 201, order-4, FP64 validation run.  A step is a few
        # microseconds, so launches and latency are what counts.
        dict(name="shot2d_f64_small", kind="shot", nx=201, nz=201, M=4, bits=64, bc="free", damp=False, nt=500, nsrc=1),
        # One ordinary 2D survey shot of odd sides with an absorbing layer.
        dict(name="shot2d_mid", kind="shot", nx=1013, nz=777, M=8, bits=32, bc="free", damp=True, nt=400, nsrc=1),
        # One large 2D shot: the wavefields are far larger than the L2.
        dict(name="shot2d_large", kind="shot", nx=8192, nz=4096, M=8, bits=32, bc="free", damp=False, nt=80, nsrc=2),
        # The 3D shot of the method's main configuration, with the table built beforehand,
        # as for every shot of a survey after the first.
        dict(name="shot3d_large", kind="shot", nx=512, ny=512, nz=384, M=8, bits=32, bc="free", damp=False, nt=80, nsrc=8),
        # A small 3D shot over a rigid surface: odd sides, order 4, absorbing layer.
        dict(name="shot3d_small", kind="shot", nx=131, ny=97, nz=110, M=4, bits=32, bc="rigid", damp=True, nt=200, nsrc=1),
        # 48 shots of uneven grids propagated together (the multi-shot forward run).
        dict(name="batch2d", kind="batch", shots=48, layout=4, lo=400, hi=1200, M=8, nt=200),
        # Inversion step over many shots: forward with checkpoints, residuals, gradients.
        dict(name="gradient_batch2d", kind="gradient", shots=24, layout=9, lo=400, hi=1200, M=8, nt=160, n_ckpt=8),
        # Inversion of one shot through torch autograd.
        dict(name="gradient_autograd2d", kind="autograd", nx=613, nz=487, M=4, nt=240, n_ckpt=6),
        # A whole staggered shot, stencils included: 1001 x 1001, order 8.
        dict(name="staggered2d_whole", kind="staggered", nx=1001, nz=1001, M=8, bc="free", nt=500, build=True),
        # A 3D staggered shot, table built beforehand.
        dict(name="staggered3d", kind="staggered", nx=160, ny=144, nz=122, M=4, bc="free", nt=60, build=False),
        # Stencils of a 3D topography and the training rows taken from them.
        dict(name="build3d", kind="build", nx=256, ny=256, nz=192, M=8, bc="free"),
        # One training step of the learned-stencil network (4 x 256) on a minibatch.
        dict(name="train_step", kind="train", width=256, layers=4, rows=40000, batch=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["shot2", "shot3", "batch", "gradient", "autograd", "staggered2", "staggered3", "build", "train"])
    bc = rng.choice(["free", "free", "rigid"])
    if kind == "shot2":
        if rng.random() < 0.3:
            n = dict(nx=_log_int(rng, 120, 640), nz=_log_int(rng, 120, 640))
            return dict(kind="shot", **n, M=rng.choice([2, 4, 6, 8]), bits=64, bc=bc, damp=rng.random() < 0.5,
                        nt=rng.randint(100, 500), nsrc=rng.randint(1, 4))
        n = dict(nx=_log_int(rng, 300, 8192), nz=_log_int(rng, 300, 4096))
        return dict(kind="shot", **n, M=rng.choice([4, 8, 8]), bits=32, bc=bc, damp=rng.random() < 0.5,
                    nt=max(40, min(500, int(2e9 / math.prod(n.values())))), nsrc=rng.randint(1, 4))
    if kind == "shot3":
        n = dict(nx=_log_int(rng, 70, 512), ny=_log_int(rng, 70, 512), nz=_log_int(rng, 80, 384))
        return dict(kind="shot", **n, M=rng.choice([4, 6, 8, 8]), bits=32, bc=bc, damp=rng.random() < 0.5,
                    nt=max(40, min(300, int(2.5e9 / math.prod(n.values())))), nsrc=rng.randint(1, 8))
    if kind in ("batch", "gradient"):
        c = dict(kind=kind, shots=rng.randint(3, 48 if kind == "batch" else 24), layout=rng.randint(0, 10 ** 6), lo=400,
                 hi=1200, M=rng.choice([4, 8, 8]), nt=rng.randint(80, 200 if kind == "batch" else 160))
        return c if kind == "batch" else dict(c, n_ckpt=rng.randint(2, 12))
    if kind == "autograd":
        return dict(kind="autograd", nx=_log_int(rng, 200, 1200), nz=_log_int(rng, 200, 1200), M=rng.choice([4, 8]),
                    nt=rng.randint(120, 240), n_ckpt=rng.randint(1, 10))
    if kind == "staggered2":
        return dict(kind="staggered", nx=_log_int(rng, 300, 1400), nz=_log_int(rng, 300, 1400), M=rng.choice([4, 8, 8]), bc=bc,
                    nt=rng.randint(120, 500), build=rng.random() < 0.5)
    if kind == "staggered3":
        return dict(kind="staggered", nx=_log_int(rng, 60, 180), ny=_log_int(rng, 60, 180), nz=_log_int(rng, 80, 140),
                    M=rng.choice([4, 4, 8]), bc="free", nt=rng.randint(30, 60), build=False)
    if kind == "build":
        if rng.random() < 0.4:
            return dict(kind="build", nx=_log_int(rng, 200, 2000), nz=_log_int(rng, 200, 1200), M=rng.choice([4, 8]), bc=bc)
        return dict(kind="build", nx=_log_int(rng, 64, 256), ny=_log_int(rng, 64, 256), nz=_log_int(rng, 80, 192),
                    M=rng.choice([4, 8, 8]), bc=bc)
    return dict(kind="train", width=rng.choice([64, 128, 256, 256]), layers=rng.randint(2, 4), rows=40000,
                batch=_log_int(rng, 512, 16384))


def _n(case):
    """Grid sizes in logical order: x, [y,] z."""
    return [case[k] for k in ("nx", "ny", "nz") if k in case]


def _row_cap(case):
    """Room for the training rows of one topography: about H rows per surface node."""
    return int(1.3 * (case["M"] // 2) * math.prod(_n(case)[:-1])) + 64


def _sides(case):
    """Grids of a batch: the case's own, the same for every seed."""
    r = random.Random(case["layout"])
    return [(r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"])) for _ in range(case["shots"])]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _surface2d(g, n, h, sinusoid):
    """(zs, dzs) of a 2D surface.  Without the sinusoid it is flat at both side edges."""
    Lx, Lz = (n[0] - 1) * h, (n[1] - 1) * h
    a = g.uniform(0.12, 0.18) * Lz + 0.37 * h
    b, lam = (g.uniform(1.0, 6.0) * h, g.uniform(80.0, 250.0) * h) if sinusoid else (0.0, h)
    k = 2 * math.pi / lam
    hills = [(g.uniform(2.0, 5.0) * h, g.uniform(0.3, 0.7) * Lx, min(g.uniform(15.0, 40.0) * h, 0.07 * Lx)) for _ in range(3)]

    def zs(x):
        z = a + b * torch.sin(k * x)
        for H, c, s in hills:
            z = z - H * torch.exp(-(x - c) ** 2 / (2 * s * s))
        return z

    def dzs(x):
        z = b * k * torch.cos(k * x)
        for H, c, s in hills:
            z = z + H * (x - c) / (s * s) * torch.exp(-(x - c) ** 2 / (2 * s * s))
        return z
    return zs, dzs


def _smooth(g, shape, cell, dev):
    """Smooth random field in [0, 1]: uniform values every `cell` nodes, interpolated."""
    coarse = [max(2, s // cell + 2) for s in shape]
    c = torch.as_tensor(g.uniform(size=coarse), dtype=torch.float32, device=dev)
    return F.interpolate(c[None, None], size=tuple(shape), mode="trilinear" if len(shape) == 3 else "bilinear",
                         align_corners=True)[0, 0]


def _model(n, h, seed, bits, nsrc, nt, rec_stride, sinusoid=True, f64_flat=False, dev=None):
    """SDF, velocity, wavelet, sources, receivers and time step of one shot."""
    dev = dev or DEV
    g = np.random.default_rng(seed)
    dt = 0.4 * h / CMAX
    d = len(n)
    ft = torch.float64 if bits == 64 else torch.float32
    if d == 2:
        if f64_flat:
            z0 = (0.2 * n[1] + g.uniform(0.1, 0.9)) * h
            zs, dzs = (lambda x: torch.full_like(x, z0)), torch.zeros_like
        else:
            zs, dzs = _surface2d(g, n, h, sinusoid)
        sdf = inputs.heightfield_sdf_2d(n[0], n[1], h, zs, dzs, device=dev)
        x = torch.arange(n[0], dtype=torch.float64) * h
        depth = zs(x)
        rx = np.arange(5, n[0] - 5, rec_stride) * h
        rec = np.stack([rx, depth.numpy()[5:n[0] - 5:rec_stride] + 2 * h], 1)
        sx = g.uniform(0.35, 0.65, nsrc) * (n[0] - 1) * h
        src = np.stack([sx, zs(torch.as_tensor(sx)).numpy() + g.uniform(8.0, 16.0, nsrc) * h], 1)
    else:
        Lx, Ly = (n[0] - 1) * h, (n[1] - 1) * h
        m = min(n)
        prm = inputs.hills_params(8, int(g.integers(1 << 30)), Lx, Ly, hmin=2.0 * h, hmax=0.12 * m * h, smin=0.12 * m * h,
                                  smax=0.4 * m * h)
        parts = inputs.hills_surface(prm, datum=(0.3 * n[2] + 0.37) * h, zmin=10 * h)
        sdf, zsurf = inputs.heightfield_sdf_3d(n[0], n[1], n[2], h, parts, device=dev)
        Y, X = np.meshgrid(np.arange(4, n[1] - 4, rec_stride), np.arange(4, n[0] - 4, rec_stride), indexing="ij")
        rec = np.stack([X.ravel() * h, Y.ravel() * h, zsurf[Y, X].ravel() + 2 * h], 1)
        ix = (g.uniform(0.35, 0.65, nsrc) * n[0]).astype(int)
        iy = (g.uniform(0.35, 0.65, nsrc) * n[1]).astype(int)
        src = np.stack([(ix + 0.3) * h, (iy + 0.6) * h, zsurf[iy, ix] + g.uniform(5.0, 9.0, nsrc) * h], 1)
    shape = tuple(reversed(n))
    span = torch.linspace(0, 1, shape[0], device=dev).reshape((-1,) + (1,) * (d - 1))
    vel = 1500.0 + 2500.0 * (0.5 * _smooth(g, shape, 50, dev) + 0.5 * span)
    f0 = min(40.0, max(10.0, 1.5 / (0.45 * nt * dt)))
    c = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)
    return dict(n=list(n), h=h, dt=dt, nt=nt, f0=f0, sdf=c(sdf), vel=vel.to(ft).contiguous(), src=c(src), rec=c(rec),
                wavelet=c(inputs.ricker(f0, dt, nt)).to(ft))


def _layer(case, h):
    return (LAYER, inputs.damping_eta(CMAX, LAYER, h, 1e-8)) if case.get("damp") else None


def _shot_model(case, seed, dev=None):
    k = case["kind"]
    if k == "shot":
        return _model(_n(case), 10.0, seed, case["bits"], case["nsrc"], case["nt"], 4, sinusoid=case["damp"],
                      f64_flat=case["bits"] == 64, dev=dev)
    if k == "autograd":
        return _model(_n(case), 10.0, seed, 32, 1, case["nt"], 4, sinusoid=False, dev=dev)
    m = _model(_n(case), 5.0, seed, 32, 1, case["nt"], 2, dev=dev)
    m["rho"] = torch.full_like(m["vel"], 1000.0)
    return m


def _batch_models(case, seed, dev=None):
    return [_model(n, 10.0, seed * 1000 + i, 32, 1, case["nt"], 4, dev=dev) for i, n in enumerate(_sides(case))]


def _observed(m):
    """Recorded data of a shot: the direct arrival of a constant medium at each receiver."""
    c = 2300.0
    dev = m["rec"].device
    r = (m["rec"] - m["src"][0]).norm(dim=1) + 50.0
    t = torch.arange(1, m["nt"] + 1, dtype=torch.float64, device=dev) * m["dt"]
    x = (math.pi * m["f0"] * (t[None] - 1.5 / m["f0"] - r[:, None] / c)) ** 2
    amp = torch.sqrt(c / (2 * r * m["f0"])) / (2 * math.pi * c * c)
    return (amp[:, None] * (1 - 2 * x) * torch.exp(-x)).float()


def _train_inputs(case, seed, dev=None):
    """Network inputs (SDF samples around seeded plane-like surfaces, flags, order), weights as targets, parameters."""
    dev = dev or DEV
    g = torch.Generator(device="cpu").manual_seed(seed)
    o = np.array([p for p in itertools.product(range(-4, 5), repeat=3) if np.dot(p, p) <= 16], dtype=np.float32)
    rows, n_in, n_out = case["rows"], len(o) + 3, 81
    nrm = torch.randn((rows, 3), generator=g).to(dev)
    nrm[:, 2] += 3.0
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    X = torch.empty((rows, n_in), dtype=torch.float32, device=dev)
    X[:, :-3] = nrm @ torch.as_tensor(o, device=dev).T + (4.0 * torch.rand((rows, 1), generator=g)).to(dev)
    X[:, -3:] = torch.tensor([1.0, 0.0, 1.0], device=dev)
    T = (0.3 * torch.randn((rows, n_out), generator=g)).to(dev)
    idx = torch.randperm(rows, generator=g)[:case["batch"]].to(dev)
    p0 = torch.as_tensor(inputs.mlp_init(n_in, case["width"], case["layers"], n_out, seed), device=dev)
    return dict(X=X.to(torch.bfloat16).contiguous(), T=T.contiguous(), idx=idx, p0=p0, n_in=n_in, n_out=n_out)


def prepare(case, seed):
    k = case["kind"]
    if k in ("shot", "autograd", "staggered"):
        m = _shot_model(case, seed)
        form = "staggered" if k == "staggered" else "second"
        if not case.get("build"):
            m["table"] = ib.ib_build_stencils(m["sdf"], m["h"], case.get("bc", "free"), form, case["M"])
        if k == "autograd":
            m["observed"] = _observed(m)
        return dict(case=case, m=m)
    if k in ("batch", "gradient"):
        ms = _batch_models(case, seed)
        tables = [ib.ib_build_stencils(m["sdf"], m["h"], "free", "second", case["M"]) for m in ms]
        damp = _layer(dict(damp=True), 10.0)
        shots = [dict(vel=m["vel"], wavelet=m["wavelet"], src=m["src"], rec=m["rec"], damp=damp) for m in ms]
        st = dict(case=case, tables=tables, shots=shots, dt=ms[0]["dt"])
        if k == "gradient":
            st["observed"] = [_observed(m) for m in ms]
            st["ckpts"] = [torch.empty(ib.ib_checkpoint_bytes(t, 32, case["nt"], case["n_ckpt"]), dtype=torch.uint8,
                                       device=DEV) for t in tables]
        return st
    if k == "build":
        m = _model(_n(case), 10.0, seed, 32, 1, 1, 4)
        net = ib.Mlp(len(_n(case)), case["M"])
        # the program gathers training rows into buffers of a fixed size
        return dict(case=case, m=m, net=net, nodes=torch.zeros(_row_cap(case), dtype=torch.int64, device=DEV),
                    weights=torch.zeros((_row_cap(case), net.n_out), device=DEV))
    t = _train_inputs(case, seed)
    return dict(case=case, t=t, net=ib.Mlp(3, 8, case["width"], case["layers"]))


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "shot":
        m = st["m"]
        return ib.ib_forward(m["table"], m["vel"], m["wavelet"], m["src"], m["rec"], m["dt"], m["nt"],
                             damp=_layer(case, m["h"]))
    if k == "staggered":
        m = st["m"]
        table = m.get("table") or ib.ib_build_stencils(m["sdf"], m["h"], case["bc"], "staggered", case["M"])
        return ib.ib_forward(table, m["vel"], m["wavelet"], m["src"], m["rec"], m["dt"], m["nt"], rho=m["rho"])
    if k == "autograd":
        m = st["m"]
        vel = m["vel"].detach().requires_grad_(True)
        traces = ib.Forward.apply(vel, m["table"], m["wavelet"], m["src"], m["rec"], m["dt"], m["nt"], case["n_ckpt"])
        loss = 0.5 * ((traces - m["observed"]) ** 2).sum()
        loss.backward()
        return traces.detach(), vel.grad
    if k == "batch":
        return ib.ib_forward_batch(st["tables"], st["shots"], st["dt"], case["nt"])
    if k == "gradient":
        traces = ib.ib_forward_batch_ckpt(st["tables"], st["shots"], st["dt"], case["nt"], st["ckpts"], case["n_ckpt"])
        res = [t - o for t, o in zip(traces, st["observed"])]
        return traces, ib.ib_adjoint_batch(st["tables"], st["shots"], st["dt"], case["nt"], st["ckpts"], case["n_ckpt"], res)
    if k == "build":
        m = st["m"]
        table = ib.ib_build_stencils(m["sdf"], m["h"], case["bc"], "second", case["M"])
        s = table.stats()
        nodes, weights = ib.ib_mlp_targets(table, st["net"])
        k = min(len(nodes), len(st["nodes"]))
        st["nodes"][:k] = nodes[:k]
        st["weights"][:k] = weights[:k]
        return dict(nodes=st["nodes"], weights=st["weights"], rows=s["rows"][0], nnz=s["nnz"][0],
                    points=s["n_boundary_points"], grown=s["n_grown"], reduced=s["n_reduced"])
    t, net = st["t"], st["net"]
    net.set_params(t["p0"])
    loss = ib.ib_mlp_train_step(net, t["X"], t["T"], t["idx"], lr=1e-3)
    return loss, net.buffers()[1].clone()   # the buffers are the network's and go with it


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _n_rec(n, stride):
    if len(n) == 2:
        return len(range(5, n[0] - 5, stride))
    return len(range(4, n[0] - 4, stride)) * len(range(4, n[1] - 4, stride))


def _fit_work(n, M, staggered):
    """Stencil construction: SDF read, about H rows per surface node (d gradients of one
    field and one coupled divergence of d fields in the staggered form); per row the Gram
    matrix of m rows and c unknowns and its factor; a support of 21 (2D) or 81 (3D) nodes."""
    d, H = len(n), M // 2
    rows = H * (n[0] if d == 2 else n[0] * n[1])
    c, sup = (15, 21) if d == 2 else (35, 81)
    one = lambda f: (f * sup + 30) * (f * c) ** 2 + (f * c) ** 3 / 3
    flops = rows * ((d * one(1) + one(d)) if staggered else one(1))
    nnz = rows * 0.8 * sup * (2 * d if staggered else 1)
    return math.prod(n) * 8 + nnz * 12, flops


def work(case):
    """Time steps: every step reads p, the previous field and the coefficient and writes the
    next field (staggered: reads and writes p and each v, reads the coefficients); the
    stencil's arithmetic.  Gradients add a recomputation and an adjoint step (read mu twice,
    K, three stored fields and the gradient, write mu and the gradient) per step."""
    k = case["kind"]
    if k in ("shot", "autograd", "staggered"):
        n, H, nt = _n(case), case["M"] // 2, case["nt"]
        d, N, es = len(n), math.prod(n), case.get("bits", 32) // 8
        io = N * es + _n_rec(n, 2 if k == "staggered" else 4) * nt * es
        if k == "staggered":
            b, f = nt * N * es * (3 + 2 * d), nt * N * (6 * d * H + 4)
            if case["build"]:
                fb, ff = _fit_work(n, case["M"], True)
                b, f = b + fb, f + ff
            return dict(bytes=b + io, flops=f)
        steps = 1 if k == "shot" else 2
        b, f = steps * nt * N * 4 * es, steps * nt * N * (4 * d * H + 6)
        if k == "autograd":
            b, f = b + nt * N * 9 * es, f + nt * N * (4 * d * H + 16)
        return dict(bytes=b + io, flops=f)
    if k in ("batch", "gradient"):
        N = sum(a * b for a, b in _sides(case))
        H, nt = case["M"] // 2, case["nt"]
        if k == "batch":
            return dict(bytes=nt * N * 16, flops=nt * N * (8 * H + 6))
        return dict(bytes=nt * N * (16 + 16 + 36), flops=nt * N * (3 * (8 * H + 6) + 10))
    if k == "build":
        b, f = _fit_work(_n(case), case["M"], False)
        return dict(bytes=b, flops=f)
    dims = [260] + [case["width"]] * case["layers"] + [81]
    w = sum(a * b for a, b in zip(dims, dims[1:]))
    r = case["batch"]
    return dict(bytes=r * (260 * 2 + 81 * 4) + w * 4 * 7, flops=2 * r * w * 3 - 2 * r * dims[0] * dims[1])


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _weights(offs, deriv):
    """Finite-difference weights at the offsets, from the Taylor system."""
    n = len(offs)
    A = np.array([[float(o) ** m / math.factorial(m) for o in offs] for m in range(n)])
    return np.linalg.solve(A, np.eye(n)[deriv])


def _poly_mul(p, q):
    out = {}
    for a, u in p.items():
        for b, v in q.items():
            s = tuple(i + j for i, j in zip(a, b))
            out[s] = out.get(s, 0.0) + u * v
    return out


def _conditions(vector, bc, d, P):
    """Boundary conditions up to order P: rows of (field, normal axis or -1, derivative, factor)."""
    e = lambda a: tuple(int(i == a) for i in range(d))
    D = lambda a: {e(a): 1.0}
    lap = {tuple(2 * i for i in e(a)): 1.0 for a in range(d)}
    L = [{(0,) * d: 1.0}]
    for _ in range(4):
        L.append(_poly_mul(L[-1], lap))
    T = lambda op, f, ax, s=1.0: [(f, ax, al, s * c) for al, c in op.items()]
    rows = []
    if not vector and bc == "free":
        rows = [T(L[k], 0, -1) for k in range(5) if 2 * k <= P]
    elif not vector:
        rows = [sum((T(_poly_mul(D(a), L[k]), 0, a) for a in range(d)), []) for k in range(5) if 2 * k + 1 <= P]
    elif bc == "free":
        rows = [sum((T(_poly_mul(D(a), L[k]), a, -1) for a in range(d)), []) for k in range(5) if 2 * k + 1 <= P]
    else:
        rows = [sum((T(L[0], a, a) for a in range(d)), [])]
        rows += [sum((T(_poly_mul(_poly_mul(D(a), D(b)), L[k]), a, b) for a in range(d) for b in range(d)), [])
                 for k in range(5) if 2 * k + 2 <= P]
        pairs = [(0, 1)] if d == 2 else [(1, 2), (2, 0), (0, 1)]
        rows += [T(_poly_mul(D(i), L[k]), j, -1) + T(_poly_mul(D(j), L[k]), i, -1, -1.0)
                 for k in range(5) if 2 * k + 1 <= P for i, j in pairs]
    return rows


def _mono(x, exps):
    """prod_a x_a^e_a / e_a! for each exponent tuple (0 where one is negative): [.., len(exps)]."""
    d = x.shape[-1]
    top = max(max(max(e) for e in exps), 0)
    pw = [torch.ones_like(x)]
    for j in range(1, top + 1):
        pw.append(pw[-1] * x / j)
    cols = []
    for e in exps:
        if min(e) < 0:
            cols.append(torch.zeros_like(x[..., 0]))
            continue
        v = pw[e[0]][..., 0]
        for a in range(1, d):
            v = v * pw[e[a]][..., a]
        cols.append(v)
    return torch.stack(cols, -1)


def _extreme(G):
    """Largest eigenvalue of each symmetric positive matrix, by repeated squaring and a Rayleigh quotient."""
    B = G / torch.linalg.matrix_norm(G)[:, None, None]
    for _ in range(11):
        B = B @ B
        B = B / torch.linalg.matrix_norm(B).clamp_min(1e-300)[:, None, None]
    x = B @ (1.0 + 0.01 * torch.arange(G.shape[-1], dtype=G.dtype, device=G.device) % 7)[None, :, None].expand(G.shape[0], -1, 1)
    return (x.mT @ (G @ x))[:, 0, 0] / (x.mT @ x)[:, 0, 0]


class _Fits:
    """Boundary points of a topography and the modified rows of its operators."""

    def __init__(self, sdf, h, M, bc):
        self.s, self.M, self.bc, self.dev = sdf / h, M, bc, sdf.device
        self.n = list(reversed(sdf.shape))
        self.d = d = len(self.n)
        self.st = [math.prod(self.n[:a]) for a in range(d)]
        self.flat = s = self.s.reshape(-1)
        lin = torch.nonzero(s.abs() <= 0.5 * math.sqrt(d))[:, 0]
        c = self._coords(lin)
        grad = torch.zeros((lin.numel(), d), dtype=torch.float64, device=self.dev)
        for a in range(d):
            room = torch.minimum(c[:, a], self.n[a] - 1 - c[:, a])
            order = torch.minimum(2 * room, torch.full_like(room, M))
            for q in range(2, M + 1, 2):
                i = torch.nonzero(order == q)[:, 0]
                w = _weights(range(-q // 2, q // 2 + 1), 1)
                for k in range(1, q // 2 + 1):
                    grad[i, a] += w[q // 2 + k] * (s[lin[i] + k * self.st[a]] - s[lin[i] - k * self.st[a]])
            for edge, lo in ((0, 0), (self.n[a] - 1, -self.st[a])):
                i = torch.nonzero((order == 0) & (c[:, a] == edge))[:, 0]
                grad[i, a] = s[lin[i] + lo + self.st[a]] - s[lin[i] + lo]
        norm = grad.norm(dim=1)
        nrm = grad / norm.clamp_min(1e-300)[:, None]
        off = -s[lin][:, None] * nrm
        ok = (norm > 0) & (off.abs().amax(1) <= 0.5)
        self.own, self.xb, self.nrm = c[ok], (c + off)[ok], nrm[ok]
        self.bp = torch.full((s.numel(),), -1, dtype=torch.int64, device=self.dev)
        self.bp[lin[ok]] = torch.arange(int(ok.sum()), device=self.dev)

    def _coords(self, lin):
        return torch.stack([(lin // self.st[a]) % self.n[a] for a in range(self.d)], 1)

    def _lin(self, c):
        return sum(c[..., a] * self.st[a] for a in range(self.d))

    def _inside(self, c):
        ok = torch.ones(c.shape[:-1], dtype=torch.bool, device=self.dev)
        for a in range(self.d):
            ok &= (c[..., a] >= 0) & (c[..., a] < self.n[a])
        return ok

    def mask(self, kind):
        """Interior nodes of p (0) or of v_a (1 + a, at j + e_a / 2)."""
        if kind == 0:
            return self.flat > 0
        ax = self.d - kind
        t = torch.cat([self.s.narrow(ax, 1, self.s.shape[ax] - 1), self.s.narrow(ax, self.s.shape[ax] - 1, 1)], ax)
        return (0.5 * (self.s + t) > 0).reshape(-1)

    def _shift(self, kind):
        return torch.tensor([0.5 * (kind == 1 + a) for a in range(self.d)], dtype=torch.float64, device=self.dev)

    def _kept(self, kind):
        """Interior nodes with no boundary point strictly inside their eta box (pressure only)."""
        m = self.mask(kind).clone()
        if kind == 0:
            eta = 0.5 if self.bc == "free" else 0.25
            for o in itertools.product((-1, 0, 1), repeat=self.d):
                c = self.own + torch.tensor(o, device=self.dev)
                hit = self._inside(c) & ((self.xb - c).abs().amax(1) < eta)
                m[self._lin(c[hit])] = False
        return m

    def rows(self, row_kind, fields, stencil):
        """Corrections of one operator: stencil = [(field, axis, k, weight)].  Returns per
        field (row, column, weight) and the accepted rows' (node, radius, order)."""
        d, dev, bc, f64 = self.d, self.dev, self.bc, torch.float64
        vector = fields[0] != 0
        kept = [self._kept(f) for f in fields]
        inter = [self.mask(f) for f in fields]
        x0s = self._shift(row_kind)
        rmask = self.mask(row_kind)
        ext = torch.zeros(self.flat.numel(), dtype=torch.bool, device=dev).reshape(self.s.shape)
        for f, a, k, _ in stencil:
            m = (~inter[f]).reshape(self.s.shape)
            ax, n = d - 1 - a, self.n[a]
            if abs(k) < n:
                ext.narrow(ax, max(0, -k), n - abs(k)).logical_or_(m.narrow(ax, max(0, k), n - abs(k)))
        left = torch.nonzero(rmask & ext.reshape(-1))[:, 0]
        out = [([], [], []) for _ in fields]
        info = []
        tol = 1e-3 if bc == "free" else 1e-2
        top = min(self.M, 4)
        for P in range(top, 1, -2):
            exps = [e for e in itertools.product(range(P + 1), repeat=d) if sum(e) <= P]
            T, nf = len(exps), len(fields)
            nc = T * nf
            cond = _conditions(vector, bc, d, P)
            ex = torch.stack([torch.tensor([k * (a == b) for b in range(d)], dtype=f64, device=dev) +
                              self._shift(fields[f]) - x0s for f, a, k, _ in stencil])
            phi_e = torch.zeros((len(stencil), nc), dtype=f64, device=dev)
            m = _mono(ex, exps)
            for i, (f, _, _, w) in enumerate(stencil):
                phi_e[i, f * T:(f + 1) * T] = w * m[i]
            for gstep in range(7):
                if not left.numel():
                    break
                r = (P + 1) / 2 + 0.5 * gstep
                R = int(math.ceil(r)) + 1
                grid = torch.tensor(list(itertools.product(range(-R, R + 1), repeat=d)), device=dev)
                ball = []
                for f in fields:
                    x = grid + self._shift(f) - x0s
                    sel = (x * x).sum(1) <= r * r + 1e-9
                    ball.append((grid[sel], _mono(x[sel], exps)))
                nsup = sum(b[0].shape[0] for b in ball)
                step = max(1, int(1.5e8 / (grid.shape[0] * (d + 2) + (nsup + 40 * len(cond)) * nc + 6 * nc * nc)))
                again = []
                for at in range(0, left.numel(), step):
                    lin = left[at:at + step]
                    c = self._coords(lin)
                    ob = c[:, None] + grid
                    ins = self._inside(ob)
                    b = torch.where(ins, self.bp[torch.where(ins, self._lin(ob), 0)], -1)
                    rel = self.xb[b.clamp_min(0)] - (c + x0s)[:, None] if self.xb.numel() else ob * 0.0
                    near = (b >= 0) & ((rel * rel).sum(-1) <= r * r + 1e-9)
                    nb = near.sum(1)
                    most = int(nb.max()) if nb.numel() else 0
                    pick = torch.argsort((~near).to(torch.int8), dim=1, stable=True)[:, :most]
                    near, b = near.gather(1, pick), b.gather(1, pick).clamp_min(0)
                    rel = rel.gather(1, pick[..., None].expand(-1, -1, d))
                    A = torch.zeros((lin.numel(), nsup + most * len(cond), nc), dtype=f64, device=dev)
                    sels, i0 = [], 0
                    for f, (o, phi) in enumerate(ball):
                        q = c[:, None] + o
                        ins = self._inside(q)
                        ql = torch.where(ins, self._lin(q), 0)
                        sel = ins & kept[f][ql]
                        A[:, i0:i0 + len(o), f * T:(f + 1) * T] = sel[..., None] * phi
                        sels.append((sel, ql, i0))
                        i0 += len(o)
                    if most:
                        nn = self.nrm[b]
                        for row in cond:
                            for f, ax, al, cf in row:
                                v = cf * _mono(rel, [tuple(i - j for i, j in zip(e, al)) for e in exps])
                                if ax >= 0:
                                    v = v * nn[..., ax:ax + 1]
                                A[:, i0:i0 + most, f * T:(f + 1) * T] += v * near[..., None]
                            i0 += most
                    count = sum(s[0].sum(1) for s in sels) + nb * len(cond)
                    G = A.mT @ A
                    chol, bad = torch.linalg.cholesky_ex(G)
                    good = torch.nonzero((bad == 0) & (count >= nc))[:, 0]
                    again_mask = torch.ones(lin.numel(), dtype=torch.bool, device=dev)
                    if good.numel():
                        A, G, chol = A[good], G[good], chol[good]
                        ratio = torch.sqrt(1.0 / (_extreme(G) * _extreme(torch.cholesky_inverse(chol))))
                        ok = torch.nonzero(ratio > tol)[:, 0]
                        good, A, chol = good[ok], A[ok], chol[ok]
                    if good.numel():
                        again_mask[good] = False
                        E = torch.zeros((good.numel(), len(stencil)), dtype=f64, device=dev)
                        for i, (f, a, k, _) in enumerate(stencil):
                            q = c[good].clone()
                            q[:, a] += k
                            ins = self._inside(q)
                            E[:, i] = (ins & ~inter[f][torch.where(ins, self._lin(q), 0)]).to(f64)
                        u = (E @ phi_e)[..., None]
                        z = torch.cholesky_solve(u, chol)
                        for _ in range(2):
                            z = z + torch.cholesky_solve(u - A.mT @ (A @ z), chol)
                        y = (A @ z)[..., 0]
                        for f, (sel, ql, i0) in enumerate(sels):
                            ri, ci = torch.nonzero(sel[good], as_tuple=True)
                            out[f][0].append(lin[good][ri])
                            out[f][1].append(ql[good][ri, ci])
                            out[f][2].append(y[:, i0:i0 + sel.shape[1]][ri, ci])
                        info.append((lin[good], torch.full_like(good, int(2 * r)), torch.full_like(good, P)))
                    again.append(lin[again_mask])
                left = torch.cat(again)
        none = torch.zeros(0, dtype=torch.int64, device=dev)
        cat = lambda v, t: torch.cat(v) if v else none.to(t)
        return ([(cat(o[0], torch.int64), cat(o[1], torch.int64), cat(o[2], f64)) for o in out],
                tuple(cat([i[j] for i in info], torch.int64) for j in range(3)))


def _laplacian_stencil(d, M):
    w = _weights(range(-(M // 2), M // 2 + 1), 2)
    return [(0, a, k, w[k + M // 2]) for a in range(d) for k in range(-(M // 2), M // 2 + 1) if k]


def _points(fits, x, h, scale):
    """Multilinear weights of points on the interior nodes: (nodes, weights), [points][2^d]."""
    xi = x / h
    base = torch.floor(xi).to(torch.int64)
    fr = xi - base
    idx, wt = [], []
    for bits in itertools.product((0, 1), repeat=fits.d):
        b = torch.tensor(bits, device=fits.dev)
        c = base + b
        w = torch.where(b == 1, fr, 1 - fr).prod(1)
        ins = fits._inside(c)
        l = torch.where(ins, fits._lin(c), 0)
        idx.append(l)
        wt.append(torch.where(ins & (fits.flat[l] > 0), w * scale, 0.0))
    return torch.stack(idx, 1), torch.stack(wt, 1)


def _exact_leapfrog(m, M, bc, damp, want_grad=None):
    """Traces of the second-order form; with want_grad (traces -> cotangent) also dJ/dvel."""
    fits = _Fits(m["sdf"], m["h"], M, bc)
    d, H, dt, h = fits.d, M // 2, m["dt"], m["h"]
    (rows, cols, w), _ = fits.rows(0, [0], _laplacian_stencil(d, M))[0][0], None
    w2 = _weights(range(-H, H + 1), 2)
    shape = m["sdf"].shape
    mask = fits.mask(0).reshape(shape)
    vel = m["vel"].double().requires_grad_(want_grad is not None)
    K = torch.where(mask, (vel * dt / h) ** 2, 0.0)
    si, sw = _points(fits, m["src"], h, dt * dt / h ** d)
    S = torch.zeros(mask.numel(), dtype=torch.float64, device=fits.dev)
    S.index_add_(0, si.reshape(-1), sw.reshape(-1))
    S = S.reshape(shape)
    ri, rw = _points(fits, m["rec"], h, 1.0)
    wav = m["wavelet"].double().cpu().tolist()
    a = None
    if damp is not None:
        W, eta = damp
        q = torch.zeros(shape, dtype=torch.float64, device=fits.dev)
        for ax in range(d):
            n = fits.n[ax]
            x = torch.arange(n, dtype=torch.float64, device=fits.dev)
            far = (x - (n - 1 - W)).clamp_min(0)
            q = q + (((W - x).clamp_min(0) + far) if ax < d - 1 else far).reshape(
                [n if j == d - 1 - ax else 1 for j in range(d)]) ** 2
        a = 0.5 * eta * dt * (q / (W * W)).clamp_max(1.0)

    def lap(p):
        pp = F.pad(p, (H, H) * d)
        out = d * w2[H] * p
        for ax in range(d):
            v = pp
            for o in range(d):
                if o != ax:
                    v = v.narrow(o, H, shape[o])
            for k in range(1, H + 1):
                out = out + w2[H + k] * (v.narrow(ax, H + k, shape[ax]) + v.narrow(ax, H - k, shape[ax]))
        return out.reshape(-1).index_add(0, rows, w * p.reshape(-1)[cols]).reshape(shape)

    p = prev = torch.zeros(shape, dtype=torch.float64, device=fits.dev)
    tr = []
    with torch.set_grad_enabled(want_grad is not None):
        for n in range(m["nt"]):
            f = K * lap(p) + wav[n] * S
            nxt = 2 * p - prev + f if a is None else (2 * p - (1 - a) * prev + f) / (1 + a)
            prev, p = p, nxt
            tr.append((p.reshape(-1)[ri] * rw).sum(1))
        traces = torch.stack(tr, 1)
        if want_grad is None:
            return traces
        grad, = torch.autograd.grad(traces, vel, want_grad(traces.detach()))
        return traces.detach(), grad


def _exact_staggered(m, M, bc):
    fits = _Fits(m["sdf"], m["h"], M, bc)
    d, H, dt, h = fits.d, M // 2, m["dt"], m["h"]
    c1 = _weights([j - (M - 1) / 2 for j in range(M)], 1)
    G = [fits.rows(1 + a, [0], [(0, a, k, c1[k + H - 1]) for k in range(-H + 1, H + 1)])[0][0] for a in range(d)]
    D = fits.rows(0, [1 + a for a in range(d)], [(a, a, k, c1[k + H]) for a in range(d) for k in range(-H, H)])[0]
    shape = m["sdf"].shape
    vel, rho = m["vel"].double(), m["rho"].double()
    kp = torch.where(fits.mask(0).reshape(shape), dt * rho * vel * vel / h, 0.0)
    bs = []
    for a in range(d):
        ax = d - 1 - a
        nb = torch.cat([rho.narrow(ax, 1, shape[ax] - 1), rho.narrow(ax, shape[ax] - 1, 1)], ax)
        bs.append(torch.where(fits.mask(1 + a).reshape(shape), dt * 0.5 * (1 / rho + 1 / nb) / h, 0.0))
    si, sw = _points(fits, m["src"], h, dt / h ** d)
    ri, rw = _points(fits, m["rec"], h, 1.0)
    wav = m["wavelet"].double().cpu().tolist()

    def diff(f, ax, lo, corr, src):
        """sum_k c_k (f[j + k - lo] - f[j - k + 1 - lo]) along array axis ax, and the corrections."""
        fp = F.pad(f, sum(((H, H) if o == ax else (0, 0) for o in reversed(range(d))), ()))
        n = shape[ax]
        out = 0.0
        for k in range(1, H + 1):
            out = out + c1[H + k - 1] * (fp.narrow(ax, H + k - lo, n) - fp.narrow(ax, H - k + 1 - lo, n))
        return out.reshape(-1).index_add_(0, corr[0], corr[2] * src.reshape(-1)[corr[1]]).reshape(shape)

    p = torch.zeros(shape, dtype=torch.float64, device=fits.dev)
    v = [torch.zeros_like(p) for _ in range(d)]
    tr = []
    for n in range(m["nt"]):
        v = [v[a] + bs[a] * diff(p, d - 1 - a, 0, G[a], p) for a in range(d)]
        p = p + kp * sum(diff(v[a], d - 1 - a, 1, D[a], v[a]) for a in range(d))
        p.reshape(-1).index_add_(0, si.reshape(-1), sw.reshape(-1) * wav[n])
        tr.append((p.reshape(-1)[ri] * rw).sum(1))
    return torch.stack(tr, 1)


def _exact_build(m, case):
    """Training rows: rows fitted at the first radius and full order, weights on the offsets
    |o| <= 2.5 (or 1.5) ordered by distance, then z, y, x."""
    fits = _Fits(m["sdf"], m["h"], case["M"], case["bc"])
    d, P = fits.d, min(case["M"], 4)
    [(rows, cols, w)], (lin, r2, order) = fits.rows(0, [0], _laplacian_stencil(d, case["M"]))
    nodes = torch.sort(lin[(r2 == P + 1) & (order == P)])[0]
    R = (P + 1) / 2
    offs = [o for o in itertools.product(range(-4, 5), repeat=d) if sum(i * i for i in o) <= R * R + 1e-9]
    offs.sort(key=lambda o: (sum(i * i for i in o), tuple(reversed(o))))
    code = {o: i for i, o in enumerate(offs)}
    lut = torch.full((9 ** d,), -1, dtype=torch.int64, device=fits.dev)
    for o, i in code.items():
        lut[sum((o[a] + 4) * 9 ** a for a in range(d))] = i
    at = torch.searchsorted(nodes, rows)
    keep = (at < nodes.numel()) & (nodes[at.clamp_max(max(nodes.numel() - 1, 0))] == rows)
    rows, cols, w, at = rows[keep], cols[keep], w[keep], at[keep]
    dc = fits._coords(cols) - fits._coords(rows)
    j = lut[sum((dc[:, a] + 4) * 9 ** a for a in range(d))]
    T = torch.zeros((_row_cap(case), len(offs)), dtype=torch.float64, device=fits.dev)
    T[at, j] = w
    return dict(nodes=None, weights=T, rows=None, nnz=None, points=None, grown=None, reduced=None)


def _exact_train(case, t):
    """Loss and gradient of the network with its bfloat16 weights and inputs, all arithmetic in 64 bits."""
    dims = [t["n_in"]] + [case["width"]] * case["layers"] + [t["n_out"]]
    at, params, x = 0, [], t["X"][t["idx"]].double()
    for i, o in zip(dims, dims[1:]):
        W = t["p0"][at:at + i * o].to(torch.bfloat16).double().reshape(o, i).requires_grad_(True)
        b = t["p0"][at + i * o:at + i * o + o].double().requires_grad_(True)
        at += i * o + o
        params += [W, b]
    for l in range(len(dims) - 1):
        x = x @ params[2 * l].T + params[2 * l + 1]
        if l + 2 < len(dims):
            x = torch.relu(x)
    loss = ((x - t["T"][t["idx"]].double()) ** 2).mean()
    return loss.detach().reshape(1), torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, params)])


def exact(case, seed):
    k = case["kind"]
    if k == "shot":
        m = _shot_model(case, seed)
        return _exact_leapfrog(m, case["M"], case["bc"], _layer(case, m["h"]))
    if k == "staggered":
        return _exact_staggered(_shot_model(case, seed), case["M"], case["bc"])
    if k == "autograd":
        m = _shot_model(case, seed)
        return _exact_leapfrog(m, case["M"], "free", None, lambda t: t - _observed(m).double())
    if k == "batch":
        return [_exact_leapfrog(m, case["M"], "free", _layer(dict(damp=True), 10.0)) for m in _batch_models(case, seed)]
    if k == "gradient":
        both = [_exact_leapfrog(m, case["M"], "free", _layer(dict(damp=True), 10.0),
                                lambda t, m=m: t - _observed(m).double()) for m in _batch_models(case, seed)]
        return [b[0] for b in both], [b[1] for b in both]
    if k == "build":
        return _exact_build(_model(_n(case), 10.0, seed, 32, 1, 1, 4), case)
    return _exact_train(case, _train_inputs(case, seed))
