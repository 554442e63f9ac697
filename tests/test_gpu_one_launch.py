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
