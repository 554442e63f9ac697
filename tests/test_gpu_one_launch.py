"""GPU: the 2D run in one cooperative launch at the edges of what it holds, and the step loop that
takes over where such a launch is refused."""
import numpy as np
import pytest
import torch

from oracle import sim
from paper_2309_03600_gb300 import inputs
from gpu_util import cuda, rel_l2

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")

# the repository's bounds against the FP64 oracle
TOL64 = 1e-12
TOL32 = 1e-5


def _shot(nx, nz, M, nt=60):
    w = inputs.workload_flat2d(nx=nx, nz=nz, nt=nt, M=M, z0_cells=10.3, f0=60.0, src_cells=(nx // 2 + 0.5, min(31.5, nz - 7.5)),
                               rec_x_cells=(4, nx - 5), rec_z_cells=13)
    w["wavelet"] = inputs.ricker(60.0, w["dt"], nt, t0=0.0)
    return w


@pytest.mark.parametrize("prec", [torch.float32, torch.float64])
def test_refused_launch(prec, monkeypatch):
    """Where the cooperative launch is refused, the forward (with and without checkpoints), the
    adjoint's recomputation, the stability estimate and the run without allocations go step by step."""
    w = _shot(129, 61, 8)
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", 8)
    args = (cuda(w["vel"], prec), cuda(w["wavelet"], prec), cuda(w["src"]), cuda(w["rec"]), w["dt"], 60)
    name = "f64" if prec == torch.float64 else "f32"
    tol = TOL64 if prec == torch.float64 else TOL32

    def all_calls():
        ck = torch.empty(ib.ib_checkpoint_bytes(t, 64 if prec == torch.float64 else 32, 60, 3), dtype=torch.uint8, device="cuda")
        out = [ib.ib_forward(t, *args, damp=(8, 60.0)), ib.ib_forward(t, *args, ckpt=ck, n_ckpt=3)]
        out.append(ib.ib_adjoint(t, *args, ck, 3, out[1])[0])
        out.append(ib.ib_stability(t, args[0], w["dt"], 200)[0])
        if prec == torch.float32:
            out.append(ib.ib_forward_noalloc(t, *args, torch.zeros_like(out[0])))
        ib.ib_sync_status()
        return [np.asarray(o.double().cpu() if torch.is_tensor(o) else o) for o in out]

    ref = all_calls()
    monkeypatch.setenv("IB_COOP", "0")
    ib.ib_profile_enable(1)
    got = all_calls()
    p = ib.ib_profile()
    ib.ib_profile_enable(0)
    # every step of the three 60-step runs, the 60 recomputed ones and the probe's 200
    # (the run without allocations in FP32 only)
    assert p["leap2d_" + name]["launches"] == (440 if prec == torch.float32 else 380)
    for a, b in zip(got, ref):
        assert np.abs(b).max() > 0 and rel_l2(a, b) < tol


def test_barrier_gives_up():
    """The grid barrier with a target that is never reached: its blocks leave after the bound, the
    host reads it, no run is reported as timed out, and the next run is right."""
    w = _shot(129, 61, 8)
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", 8)
    args = (cuda(w["vel"]), cuda(w["wavelet"]), cuda(w["src"]), cuda(w["rec"]), w["dt"], 60)
    ref = ib.ib_forward(t, *args)
    assert ib.ib_selftest_bounded_wait() == ib.IB_ERR_TIMEOUT
    assert "grid barrier" in ib.ib_last_error()
    assert ib.ib_sync_status() == ib.IB_OK
    assert torch.equal(ib.ib_forward(t, *args), ref)


def _both(w, t, prec, nt, monkeypatch, **kw):
    """The traces of the run in one launch, and of bursts launch by launch (held to the oracle elsewhere)."""
    args = (t, cuda(w["vel"], prec), cuda(w["wavelet"], prec), cuda(w["src"]), cuda(w["rec"]), w["dt"], nt)
    ib.ib_profile_enable(1)
    a = ib.ib_forward(*args, **kw).double().cpu().numpy()
    assert any(k.startswith("leap2d_run") for k in ib.ib_profile())
    ib.ib_profile_enable(0)
    monkeypatch.setenv("IB_STRIP", "0")
    b = ib.ib_forward(*args, **kw).double().cpu().numpy()
    ib.ib_sync_status()
    assert np.abs(b[:, -1]).max() > 0
    return a, b


@pytest.mark.parametrize("nx,nz,M,damped", [(501, 403, 2, True), (499, 402, 4, False)])
def test_four_points_a_thread_vs_oracle(nx, nz, M, damped, monkeypatch):
    """FP32 grids beyond one point a thread."""
    w, damp = _shot(nx, nz, M), ((12, 80.0) if damped else None)
    ref = sim.Leapfrog(w["sdf"], w["vel"], w["h"], M, "free", w["dt"], w["src"], w["rec"], damp=damp).forward(w["wavelet"], 60)
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", M)
    a, b = _both(w, t, torch.float32, 60, monkeypatch, damp=damp)
    assert rel_l2(a, ref) < TOL32 and rel_l2(b, ref) < TOL32


@pytest.mark.parametrize("nx,nz,M,damped", [(601, 590, 8, True), (431, 777, 6, True)])
def test_four_points_a_thread(nx, nz, M, damped, monkeypatch):
    w = _shot(nx, nz, M)
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", M)
    a, b = _both(w, t, torch.float32, 60, monkeypatch, damp=(12, 80.0) if damped else None)
    assert rel_l2(a, b) < TOL32


@pytest.mark.parametrize("nx,nz,M,amp,wave,prec", [(2600, 40, 8, 2.2, 23.0, torch.float32),
                                                   (2503, 30, 8, 2.2, 23.0, torch.float32),
                                                   (4801, 29, 4, 3.0, 15.0, torch.float64)])
def test_more_rows_than_a_block_holds(nx, nz, M, amp, wave, prec, monkeypatch):
    """Wide shallow grids over a rough surface: more than 64 rows for every block a GPU of 152
    SMs can have."""
    w = _shot(nx, nz, M)
    w["sdf"] = inputs.sinusoid_sdf(nx, nz, w["h"], z0=9.3 * w["h"], amp=amp * w["h"], wavelength=wave * w["h"])
    w["src"][:, 1] = 20.5 * w["h"]
    w["rec"][:, 1] = 14 * w["h"]
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", M)
    assert t.stats()["rows"][0] > 64 * 152
    a, b = _both(w, t, prec, 40, monkeypatch)
    assert rel_l2(a, b) < (TOL64 if prec == torch.float64 else TOL32)
