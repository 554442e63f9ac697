"""GPU: options of the construction away from their defaults, against the oracle's fits."""
import pytest

from oracle import stencils
from gpu_util import compare_tables, cuda, gpu_rows, small_hills

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")


def test_first_radius_below_one_node():
    """Every row grows from a support of its own node: the room for the entries does not
    follow from the first radius."""
    sdf, _ = small_hills(nx=14, ny=13, nz=26)
    orc = stencils.laplacian_rows(stencils.Geometry(sdf, 10.0, 4), "free", stencils.Opts(4, radius=0.5))
    o = ib.ib_opts_default(4)
    o.radius = 0.5
    t = ib.ib_build_stencils(cuda(sdf), 10.0, "free", "second", 4, opts=o)
    st = t.stats()
    assert st["n_grown"] == st["rows"][0] and st["nnz"][0] > 16 * max(st["rows"][0], 1024)
    compare_tables(orc, gpu_rows(t.export(0), sdf.shape))
