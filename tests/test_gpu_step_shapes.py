"""GPU: the shapes of the 2D steps inside the adjoint -- the recomputation launch by launch, and
every batch shape on its segment fields -- at the odd sizes of the step tests, with three
checkpoints, against the oracle's adjoint."""
import numpy as np
import pytest
import torch

from oracle import sim
from gpu_util import cuda, rel_l2
from test_gpu_leap2d import SIZES, TOL32, TOL64, _shot

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")


@pytest.mark.parametrize("nx,nz,M,damped", SIZES)
def test_recomputation_vs_oracle(nx, nz, M, damped, monkeypatch):
    w, damp = _shot(nx, nz, M, damped)
    s = sim.Leapfrog(w["sdf"], w["vel"], w["h"], M, "free", w["dt"], w["src"], w["rec"], damp=damp)
    tr, hist = s.forward(w["wavelet"], 60, keep_history=True)
    res = np.random.default_rng(3).normal(size=tr.shape)
    ref = np.ravel(s.adjoint(res, hist)[0])
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", M)
    src, rec, dt = cuda(w["src"]), cuda(w["rec"]), w["dt"]

    # one shot, launch by launch: FP64 forward with checkpoints and recomputation; FP32 likewise
    for prec, bits, ttol, gtol in ((torch.float64, 64, TOL64, TOL64 * 10), (torch.float32, 32, TOL32, TOL32)):
        vel, wv = cuda(w["vel"], prec), cuda(w["wavelet"], prec)
        for strip in ("0", "1"):
            monkeypatch.setenv("IB_STRIP", strip)
            ib.ib_profile_enable(1)
            ck = torch.empty(ib.ib_checkpoint_bytes(t, bits, 60, 3), dtype=torch.uint8, device="cuda")
            got = ib.ib_forward(t, vel, wv, src, rec, dt, 60, ckpt=ck, n_ckpt=3, damp=damp)
            g, _ = ib.ib_adjoint(t, vel, wv, src, rec, dt, 60, ck, 3, cuda(res, prec), damp=damp)
            p = ib.ib_profile()
            ib.ib_profile_enable(0)
            assert not any("run" in k for k in p)
            assert sum(p[k]["launches"] for k in p if k.startswith("leap2d")) == 120
            assert rel_l2(got.double().cpu().numpy(), tr) < ttol, (prec, strip)
            assert rel_l2(g.double().cpu().numpy().ravel(), ref) < gtol, (prec, strip)
    monkeypatch.delenv("IB_STRIP")

    # the batched recomputation in every shape
    shot = dict(vel=cuda(w["vel"], torch.float32), wavelet=cuda(w["wavelet"], torch.float32), src=src, rec=rec, damp=damp)
    ck = torch.empty(ib.ib_checkpoint_bytes(t, 32, 60, 3), dtype=torch.uint8, device="cuda")
    ib.ib_forward_batch_ckpt([t], [shot], dt, 60, [ck], 3)
    for shape in range(10):
        monkeypatch.setenv("IB_BATCH_SHAPE", str(shape))
        g, = ib.ib_adjoint_batch([t], [shot], dt, 60, [ck], 3, [cuda(res, torch.float32)])
        assert rel_l2(g.double().cpu().numpy().ravel(), ref) < TOL32, shape
    monkeypatch.setenv("IB_BATCH_SHAPE", "10")
    with pytest.raises(ib.IbError) as e:
        ib.ib_adjoint_batch([t], [shot], dt, 60, [ck], 3, [cuda(res, torch.float32)])
    assert e.value.status == ib.IB_ERR_ARG
    ib.ib_sync_status()
