"""Edges of the one-warp row fit: chunk remainders of the boundary points, supports beyond
its buffers (left to the block-per-row kernel), and rows whose support grows, against the
oracle's fits of the same rows."""
import numpy as np
import pytest

from oracle import stencils
from paper_2309_03600_gb300 import inputs
from gpu_util import compare_tables, cuda, gpu_rows

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")


def _plane(n, slope):
    """SDF of the plane through the grid's centre with normal ~ (slope, 0.7 slope, 1)."""
    nrm = np.array([slope, 0.7 * slope, 1.0])
    nrm /= np.linalg.norm(nrm)
    z, y, x = np.meshgrid(*[np.arange(k, dtype=np.float64) for k in reversed(n)], indexing="ij")
    return 10.0 * ((x - 0.47 * n[0]) * nrm[0] + (y - 0.53 * n[1]) * nrm[1] + (z - 0.44 * n[2]) * nrm[2])


# radius 2.5: 81 offsets (the default); 3.5: 179; 4.5: 389, beyond the 320 nodes a warp holds.
# slope 0 / 1: 21 / up to 36 boundary points in reach of a row at radius 2.5.
# Tolerance: that of the other table tests, (1e-8 + 1e-13 cond) of the row's largest weight.
@pytest.mark.parametrize("bc,M,radius,slope", [("free", 2, 0.0, 0.3), ("rigid", 4, 0.0, 1.0), ("free", 4, 3.5, 0.4),
                                               ("rigid", 4, 4.5, 0.6)])
def test_rows_3d(bc, M, radius, slope):
    sdf = _plane((15, 13, 14), slope)
    geom = stencils.Geometry(sdf, 10.0, M)
    orc = stencils.laplacian_rows(geom, bc, stencils.Opts(M, radius=radius))
    o = ib.ib_opts_default(M)
    o.radius = radius
    t = ib.ib_build_stencils(cuda(sdf), 10.0, bc, "second", M, opts=o)
    assert len(orc) > 100
    compare_tables(orc, gpu_rows(t.export(0), sdf.shape))


@pytest.mark.parametrize("M", [2, 4, 6, 8])
def test_rows_2d_grown(M):
    """A trough narrower than the first support: rows on its sides grow or drop an order."""
    x = np.arange(40, dtype=np.float64)[None, :]
    z = np.arange(34, dtype=np.float64)[:, None]
    sdf = 10.0 * (np.abs(x - 19.3) + 0.6 * (z - 20.2) - 1.9)
    sdf = np.maximum(sdf, 10.0 * (z - 26.4))
    geom = stencils.Geometry(sdf, 10.0, M)
    orc = stencils.laplacian_rows(geom, "free", stencils.Opts(M))
    t = ib.ib_build_stencils(cuda(sdf), 10.0, "free", "second", M)
    compare_tables(orc, gpu_rows(t.export(0), sdf.shape))
    st = t.stats()
    assert M == 2 or st["n_grown"] + st["n_reduced"] > 0
