"""GPU: a construction on a non-blocking side stream gives the table of the default stream."""
import numpy as np
import pytest
import torch

from gpu_util import cuda, small_hills

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")


@pytest.mark.parametrize("form", ["second", "staggered"])
def test_build_on_side_streams(form):
    sdf = cuda(small_hills(nx=30, ny=28, nz=26)[0])
    t = ib.ib_build_stencils(sdf, 10.0, "free", form, 4)
    n = t.stats()["n_ops"]
    ref = [t.export(i) for i in range(n)]
    torch.cuda.synchronize()
    for _ in range(4):
        s = torch.cuda.Stream()
        t = ib.ib_build_stencils(sdf, 10.0, "free", form, 4, stream=s)
        for i in range(n):
            e = t.export(i)
            assert all(np.array_equal(e[k], ref[i][k]) for k in ref[i]), i
