"""GPU: the staggered steps at the edges of their blocks.  FP32 threads own four adjacent nodes
and FP64 threads two, so the two split a row differently; FP64 is held to the oracle elsewhere
(1e-12), and FP32 has to agree with it to the repository's FP32 bound."""
import numpy as np
import pytest
import torch

from paper_2309_03600_gb300 import inputs
from gpu_util import cuda, rel_l2, small_hills

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")

TOL32 = 1e-5


def _both(t, vel, wv, src, rec, dt, nt, rho):
    out = [ib.ib_forward(t, cuda(vel, d), cuda(wv, d), cuda(src), cuda(rec), dt, nt, rho=cuda(rho, d)).double().cpu().numpy()
           for d in (torch.float64, torch.float32)]
    ib.ib_sync_status()
    return out


@pytest.mark.parametrize("nx,ny,nz,M", [(133, 17, 26, 2), (64, 25, 27, 4)])
def test_staggered3d_blocks(nx, ny, nz, M):
    sdf, zs = small_hills(nx=nx, ny=ny, nz=nz)
    h, nt = 10.0, 50
    dt = 0.3 * h / 1800.0
    # off the grid, over the edge of a block of 64 nodes where the grid has one
    src = np.array([[(63.5 if nx > 80 else nx // 2 + 0.5) * h, 7.5 * h, (nz - 7.5) * h]])
    rec = np.array([[x * h, y * h, zs[y, x] + 2 * h] for x in range(2, nx - 2, 7) for y in range(2, ny - 2, 5)])
    t = ib.ib_build_stencils(cuda(sdf), h, "free", "staggered", M)
    a, b = _both(t, np.full(sdf.shape, 1800.0), inputs.ricker(60.0, dt, nt, t0=0.0), src, rec, dt, nt,
                 np.full(sdf.shape, 1000.0))
    assert np.abs(a[:, -1]).max() > 0
    assert rel_l2(b, a) < TOL32
