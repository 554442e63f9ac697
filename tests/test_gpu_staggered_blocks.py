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


@pytest.mark.parametrize("nx,nz,M", [(127, 65, 8), (129, 64, 8), (133, 71, 2), (260, 73, 6)])
def test_staggered2d_blocks(nx, nz, M):
    h, nt = 5.0, 60
    sdf = inputs.flat_surface_sdf((nx, nz), h, 10.3 * h)
    dt = 0.4 * h / 1500.0
    # off the grid, over the corner of a block of 128 x 8 (FP32) or 64 x 8 (FP64) nodes
    src = np.array([[min(127.5, nx - 9.5) * h, 31.5 * h]])
    rec = np.array([[x * h, z * h] for x in range(3, nx - 3, 4) for z in (12, nz - 6)])
    t = ib.ib_build_stencils(cuda(sdf), h, "free", "staggered", M)
    a, b = _both(t, np.full(sdf.shape, 1500.0), inputs.ricker(100.0, dt, nt, t0=0.0), src, rec, dt, nt,
                 np.full(sdf.shape, 1000.0))
    assert np.abs(a[:, -1]).max() > 0
    assert rel_l2(b, a) < TOL32
