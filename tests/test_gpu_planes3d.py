"""GPU: the planes per block of the FP32 3D step, chosen by the grid's size, do not change a
bit of the traces."""
import numpy as np
import pytest
import torch

from paper_2309_03600_gb300 import inputs
from gpu_util import cuda, small_hills

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")


@pytest.mark.parametrize("nx,ny,nz,M", [(70, 19, 27, 8), (30, 33, 34, 4)])
def test_planes_per_block(nx, ny, nz, M, monkeypatch):
    sdf, zs = small_hills(nx=nx, ny=ny, nz=nz)
    h, nt = 10.0, 40
    dt = 0.4 * h / 1800.0
    src = cuda(np.array([[nx // 2 * h, ny // 2 * h, (nz - 7) * h]]))
    rec = cuda(np.array([[x * h, y * h, zs[y, x] + 2 * h] for x in range(2, nx - 2, 6) for y in range(2, ny - 2, 5)]))
    t = ib.ib_build_stencils(cuda(sdf), h, "free", "second", M)
    args = (t, cuda(np.full(sdf.shape, 1800.0), torch.float32), cuda(inputs.ricker(60.0, dt, nt, t0=0.0), torch.float32),
            src, rec, dt, nt)
    ref = ib.ib_forward(*args, damp=(4, 60.0))
    assert float(ref.abs().max()) > 0
    for planes in ("4", "6", "32", "96"):
        monkeypatch.setenv("IB_ZCHUNK", planes)
        assert torch.equal(ib.ib_forward(*args, damp=(4, 60.0)), ref), planes
    ib.ib_sync_status()
