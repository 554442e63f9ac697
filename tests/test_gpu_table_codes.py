"""GPU: the entry codes and offsets that the 3D steps read -- there from a table's first use, in
whatever stream or capture that falls, for supports wider than a 16-bit code can name, and in 64
bits."""
import numpy as np
import pytest
import torch

from oracle import operators, propagate, sim, stencils
from paper_2309_03600_gb300 import inputs
from gpu_util import cuda, gpu_rows, rel_l2, small_hills

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")

TOL64 = 1e-12     # the repository's bounds against FP64
TOL32 = 1e-5


def _hills(form, prec=torch.float32):
    """A fresh table and the arguments of one shot on it."""
    sdf, zs = small_hills(nx=30, ny=28, nz=26)
    h, nt = 10.0, 40
    dt = 0.3 * h / 1800.0
    src = np.array([[15 * h, 14 * h, 19 * h]])
    rec = np.array([[x * h, y * h, zs[y, x] + 2 * h] for x in range(3, 27, 4) for y in range(3, 25, 4)])
    t = ib.ib_build_stencils(cuda(sdf), h, "free", form, 4)
    args = (cuda(np.full(sdf.shape, 1800.0), prec), cuda(inputs.ricker(60.0, dt, nt, t0=0.0), prec), cuda(src), cuda(rec), dt, nt)
    rho = cuda(np.full(sdf.shape, 1000.0), prec) if form == "staggered" else None
    return t, args, rho


def test_first_staggered_run_in_a_capture():
    """A 3D staggered shot only enqueues, also the first one on its table."""
    t, args, rho = _hills("staggered")
    ref = ib.ib_forward(t, *args, rho=rho)          # and the kernels are loaded
    t, args, rho = _hills("staggered")
    out = torch.zeros_like(ref)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        g.capture_begin()
        try:
            ib.ib_forward(t, *args, rho=rho, traces=out)
        finally:
            g.capture_end()
    g.replay()
    torch.cuda.synchronize()
    assert float(ref.abs().max()) > 0 and torch.equal(out, ref)


@pytest.mark.parametrize("form", ["staggered", "second"])
def test_first_runs_on_two_streams(form):
    """The first two shots on a table, enqueued one after the other on two streams."""
    t, args, rho = _hills(form)
    ref = ib.ib_forward(t, *args, rho=rho)
    t, args, rho = _hills(form)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    out = [torch.zeros_like(ref) for _ in streams]
    torch.cuda.synchronize()
    for s, o in zip(streams, out):
        ib.ib_forward(t, *args, rho=rho, traces=o, stream=s)
    torch.cuda.synchronize()
    for o in out:
        assert torch.equal(o, ref)


def _wide(form):
    """A thin slab whose supports reach 16 or 17 nodes along x, the table, and its rows on the host."""
    h, M, n = 10.0, 2, (44, 3, 7)
    sdf = inputs.flat_surface_sdf(n, h, 2.3 * h)
    o = ib.ib_opts_default(M)
    o.radius, o.growth, o.rank_tol = 17.0, 0.0, 1e-9
    t = ib.ib_build_stencils(cuda(sdf), h, "free", form, M, opts=o, allow_rank_failure=True)
    shape = sdf.shape
    rows = [gpu_rows(t.export(i), shape) for i in range(t.stats()["n_ops"])]
    assert max(abs(o[0]) for r in rows for w, _ in r.values() for o in w) >= 16
    dt = 0.3 * h / 1800.0
    src, rec = np.array([[22 * h, h, 4 * h]]), np.array([[x * h, h, 3 * h] for x in range(3, 41, 3)])
    return t, rows, sdf, h, M, dt, src, rec, inputs.ricker(60.0, dt, 40, t0=0.0)


def test_wide_supports_staggered():
    t, rows, sdf, h, M, dt, src, rec, wv = _wide("staggered")
    geom = stencils.Geometry(sdf, h, M)
    div = {}
    for a in range(3):
        for node, (w, info) in rows[3 + a].items():
            div.setdefault(node, ({}, info))[0].update({(a,) + o: v for o, v in w.items()})
    G, D, _, _ = operators.staggered_matrices(geom, "free", stencils.Opts(M), grad_rows=rows[:3], div_rows=div)
    one = np.full(sdf.shape, 1.0)
    bv, kp = propagate.staggered_coefficients(geom, 1800.0 * one, 1000.0 * one, dt)
    S = propagate.multilinear_matrix(src, h, sdf.shape, geom.mask).toarray().sum(0) * dt / h ** 3
    ref = propagate.forward_staggered(G, D, bv, kp, S, wv, propagate.multilinear_matrix(rec, h, sdf.shape, geom.mask), 40)
    assert np.abs(ref[:, -1]).max() > 0
    for prec, tol in ((torch.float64, TOL64), (torch.float32, TOL32)):
        tr = ib.ib_forward(t, cuda(1800.0 * one, prec), cuda(wv, prec), cuda(src), cuda(rec), dt, 40, rho=cuda(1000.0 * one, prec))
        assert rel_l2(tr.double().cpu().numpy(), ref) < tol, prec
    ib.ib_sync_status()


def test_wide_supports_second_order():
    t, rows, sdf, h, M, dt, src, rec, wv = _wide("second")
    s = object.__new__(sim.Leapfrog)
    geom = stencils.Geometry(sdf, h, M)
    s.L, _ = operators.laplacian_matrix(geom, "free", stencils.Opts(M), ib_rows=rows[0])
    vel = np.full(sdf.shape, 1800.0)
    s.K = propagate.leapfrog_coefficient(vel, dt, geom.mask)
    s.S = propagate.multilinear_matrix(src, h, sdf.shape, geom.mask).toarray().sum(0) * dt * dt / h ** 3
    s.R, s.a = propagate.multilinear_matrix(rec, h, sdf.shape, geom.mask), None
    ref = s.forward(wv, 40)
    assert np.abs(ref[:, -1]).max() > 0
    for prec, tol in ((torch.float64, TOL64), (torch.float32, TOL32)):
        tr = ib.ib_forward(t, cuda(vel, prec), cuda(wv, prec), cuda(src), cuda(rec), dt, 40)
        assert rel_l2(tr.double().cpu().numpy(), ref) < tol, prec
    ib.ib_sync_status()


@pytest.mark.parametrize("n,M", [((30, 28, 26), 2), ((30, 28, 26), 6), ((70, 25, 30), 8), ((88, 84, 30), 8)])
def test_staggered_rows_in_launches_of_their_own(n, M, monkeypatch):
    """Rows with 64-bit offsets, in launches of their own, against the default: in one launch with
    the columns on the small grids, in launches of their own from 24 000 divergence rows on."""
    sdf, zs = small_hills(nx=n[0], ny=n[1], nz=n[2])
    h, nt = 10.0, 40
    dt = 0.3 * h / 1800.0
    src = np.array([[(n[0] // 2 + 0.5) * h, n[1] // 2 * h, (n[2] - 7) * h]])
    rec = np.array([[x * h, y * h, zs[y, x] + 2 * h] for x in range(3, n[0] - 3, 4) for y in range(3, n[1] - 3, 4)])
    t = ib.ib_build_stencils(cuda(sdf), h, "free", "staggered", M, allow_rank_failure=True)
    assert (t.stats()["rows"][3] >= 24000) == (n[1] == 84)
    for prec, tol in ((torch.float64, TOL64), (torch.float32, TOL32)):
        args = (t, cuda(np.full(sdf.shape, 1800.0), prec), cuda(inputs.ricker(60.0, dt, nt, t0=0.0), prec), cuda(src), cuda(rec), dt, nt)
        rho = cuda(np.full(sdf.shape, 1000.0), prec)
        monkeypatch.delenv("IB_ROW_OFF64", raising=False)
        a = ib.ib_forward(*args, rho=rho).double().cpu().numpy()
        monkeypatch.setenv("IB_ROW_OFF64", "1")
        b = ib.ib_forward(*args, rho=rho).double().cpu().numpy()
        assert np.abs(a[:, -1]).max() > 0 and rel_l2(b, a) < tol, prec
    ib.ib_sync_status()
