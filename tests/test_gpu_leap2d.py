"""GPU: the 2D leapfrog and adjoint kernels at the edges of their column and row
splits: one burst of rows per thread, marching columns of 128 nodes, and the kernel
that runs a whole shot, with immersed-boundary rows, sources and the absorbing layer
on the seams."""
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


def _shot(nx, nz, M, damped):
    """Flat surface off the grid; a source whose spread straddles node (128, 32) where the
    grid has it, receivers on the rows next to the surface and at both sides."""
    w = inputs.workload_flat2d(nx=nx, nz=nz, nt=60, M=M, z0_cells=10.3, f0=60.0,
                               src_cells=(min(127.5, nx - 8.5), min(31.5, nz - 9.5)),
                               rec_x_cells=(4, nx - 5), rec_z_cells=13)
    w["wavelet"] = inputs.ricker(60.0, w["dt"], 60, t0=0.0)
    return w, ((6, 80.0) if damped else None)


SIZES = [(127, 41, 8, False), (128, 48, 8, True), (129, 49, 8, False), (260, 37, 4, True), (133, 65, 2, False),
         (257, 130, 6, True)]


@pytest.mark.parametrize("nx,nz,M,damped", SIZES)
def test_step_kernels_vs_oracle(nx, nz, M, damped, monkeypatch):
    w, damp = _shot(nx, nz, M, damped)
    ref = sim.Leapfrog(w["sdf"], w["vel"], w["h"], M, "free", w["dt"], w["src"], w["rec"],
                       damp=damp).forward(w["wavelet"], 60)
    assert np.abs(ref[:, -1]).max() > 0
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", M)

    def run(dt_):
        return ib.ib_forward(t, cuda(w["vel"], dt_), cuda(w["wavelet"], dt_), cuda(w["src"]), cuda(w["rec"]), w["dt"],
                             60, damp=damp).double().cpu().numpy()

    assert rel_l2(run(torch.float64), ref) < TOL64
    assert rel_l2(run(torch.float32), ref) < TOL32          # the whole shot in one kernel
    for strip in ("0", "1"):
        monkeypatch.setenv("IB_STRIP", strip)
        assert rel_l2(run(torch.float32), ref) < TOL32, strip
    monkeypatch.delenv("IB_STRIP")
    shot = dict(vel=cuda(w["vel"], torch.float32), wavelet=cuda(w["wavelet"], torch.float32), src=cuda(w["src"]),
                rec=cuda(w["rec"]), damp=damp)
    for shape in range(10):
        monkeypatch.setenv("IB_BATCH_SHAPE", str(shape))
        tr, = ib.ib_forward_batch([t], [shot], w["dt"], 60)
        assert rel_l2(tr.double().cpu().numpy(), ref) < TOL32, shape
    ib.ib_sync_status()


@pytest.mark.parametrize("nx,nz,M,damped", SIZES)
def test_adjoint_kernels_vs_oracle(nx, nz, M, damped, monkeypatch):
    """Both splits of the FP32 adjoint step, single and batched, and the FP64 one, with three
    checkpoints: gradients of random residuals against the oracle's adjoint."""
    w, damp = _shot(nx, nz, M, damped)
    s = sim.Leapfrog(w["sdf"], w["vel"], w["h"], M, "free", w["dt"], w["src"], w["rec"], damp=damp)
    tr, hist = s.forward(w["wavelet"], 60, keep_history=True)
    res = np.random.default_rng(3).normal(size=tr.shape)
    ref = np.ravel(s.adjoint(res, hist)[0])
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", M)

    def grad(dt_):
        vel, wv, r = cuda(w["vel"], dt_), cuda(w["wavelet"], dt_), cuda(res, dt_)
        ck = torch.empty(ib.ib_checkpoint_bytes(t, 64 if dt_ == torch.float64 else 32, 60, 3), dtype=torch.uint8,
                         device="cuda")
        ib.ib_forward(t, vel, wv, cuda(w["src"]), cuda(w["rec"]), w["dt"], 60, ckpt=ck, n_ckpt=3, damp=damp)
        return ib.ib_adjoint(t, vel, wv, cuda(w["src"]), cuda(w["rec"]), w["dt"], 60, ck, 3, r,
                             damp=damp)[0].double().cpu().numpy().ravel()

    assert rel_l2(grad(torch.float64), ref) < TOL64 * 10
    shot = dict(vel=cuda(w["vel"], torch.float32), wavelet=cuda(w["wavelet"], torch.float32), src=cuda(w["src"]),
                rec=cuda(w["rec"]), damp=damp)
    for strip in ("0", "1"):
        monkeypatch.setenv("IB_STRIP", strip)
        assert rel_l2(grad(torch.float32), ref) < TOL32, strip
        ck = torch.empty(ib.ib_checkpoint_bytes(t, 32, 60, 3), dtype=torch.uint8, device="cuda")
        ib.ib_forward_batch_ckpt([t], [shot], w["dt"], 60, [ck], 3)
        g, = ib.ib_adjoint_batch([t], [shot], w["dt"], 60, [ck], 3, [cuda(res, torch.float32)])
        assert rel_l2(g.double().cpu().numpy().ravel(), ref) < TOL32, strip
    ib.ib_sync_status()
