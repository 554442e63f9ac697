"""GPU: inputs at the edge of what the time steps accept -- NaN velocities, wavelets that are
not finite, negative densities.  Each touches the nodes it belongs to and no others."""
import numpy as np
import pytest
import torch

from paper_2309_03600_gb300 import inputs
from gpu_util import cuda, small_hills

pytestmark = pytest.mark.gpu

ib = pytest.importorskip("paper_2309_03600_gb300.ib")


def _flat(nx=161, nz=71, nt=60, M=8):
    w = inputs.workload_flat2d(nx=nx, nz=nz, nt=nt, M=M, z0_cells=10.3, f0=60.0, src_cells=(nx // 2 + 0.5, 31.5),
                               rec_x_cells=(4, nx - 5), rec_z_cells=13)
    w["wavelet"] = inputs.ricker(60.0, w["dt"], nt, t0=0.0)
    return w


@pytest.mark.parametrize("prec", [torch.float32, torch.float64])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("strip", [None, "0", "1"])
def test_nan_velocity_is_reported(prec, sign, strip, monkeypatch):
    """A NaN of either sign in the velocity, away from the surface, makes the run's field NaN."""
    if strip:
        monkeypatch.setenv("IB_STRIP", strip)
    w = _flat()
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", 8)
    vel = cuda(w["vel"], prec)
    vel[40, 30] = torch.copysign(torch.tensor(float("nan"), dtype=prec), torch.tensor(sign, dtype=prec))
    ib.ib_forward(t, vel, cuda(w["wavelet"], prec), cuda(w["src"]), cuda(w["rec"]), w["dt"], 60)
    with pytest.raises(ib.IbError) as e:
        ib.ib_sync_status()
    assert e.value.status == ib.IB_ERR_UNSTABLE
    ib.ib_sync_status()


def _last_sample(run, wavelet, bad):
    """Traces with the last wavelet sample zero, and not finite."""
    out = []
    for v in (0.0, bad):
        wv = wavelet.copy()
        wv[-1] = v
        out.append(run(wv).double().cpu().numpy())
    try:
        ib.ib_sync_status()      # the final field holds what the source put there
    except ib.IbError as e:
        assert e.status == ib.IB_ERR_UNSTABLE
    return out


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("prec,strip,damped", [(torch.float64, None, True), (torch.float64, "0", True), (torch.float32, None, True),
                                               (torch.float32, "0", True), (torch.float32, "1", True), (torch.float32, "batch", True)])
def test_nonfinite_wavelet_stays_at_the_source_2d(prec, strip, damped, bad, monkeypatch):
    """The last sample enters the last field at the source's nodes only, so the receivers,
    none of which touches them, do not see it."""
    w = _flat()
    damp = (12, 80.0) if damped else None
    # receivers next to the source too, one node further than its spread
    near = w["src"][0] + w["h"] * np.array([[2.5, 0.0], [-2.5, 0.0], [0.0, 2.5], [1.0, -2.5]])
    w["rec"] = np.concatenate([w["rec"], near])
    t = ib.ib_build_stencils(cuda(w["sdf"]), w["h"], "free", "second", 8)
    vel, src, rec = cuda(w["vel"], prec), cuda(w["src"]), cuda(w["rec"])

    def run(wv):
        if strip == "batch":
            return ib.ib_forward_batch([t], [dict(vel=vel, wavelet=cuda(wv, prec), src=src, rec=rec, damp=damp)], w["dt"], 60)[0]
        return ib.ib_forward(t, vel, cuda(wv, prec), src, rec, w["dt"], 60, damp=damp)

    if strip in ("0", "1"):
        monkeypatch.setenv("IB_STRIP", strip)
    a, b = _last_sample(run, w["wavelet"], bad)
    assert np.abs(a[:, -1]).max() > 0
    assert np.isfinite(b).all() and np.array_equal(a, b)


@pytest.mark.parametrize("prec", [torch.float32, torch.float64])
@pytest.mark.parametrize("ndim", [2, 3])
def test_nonfinite_wavelet_stays_at_the_source_staggered(ndim, prec):
    h = 5.0
    if ndim == 2:
        sdf = inputs.flat_surface_sdf((129, 64), h, 10.3 * h)
        src = np.array([[64.5 * h, 31.5 * h]])
        rec = np.array([[x * h, z * h] for x in range(3, 126, 4) for z in (12, 58)] + [[67 * h, 31 * h], [64 * h, 34 * h]])
    else:
        sdf, zs = small_hills(h=h)
        src = np.array([[20.5 * h, 17.5 * h, 27.5 * h]])
        rec = np.array([[x * h, y * h, zs[y, x] + 2 * h] for x in range(4, 36, 5) for y in range(4, 32, 5)]
                       + [[23 * h, 17 * h, 27 * h], [20 * h, 17 * h, 30 * h]])
    dt = 0.3 * h / 1800.0
    t = ib.ib_build_stencils(cuda(sdf), h, "free", "staggered", 4)
    vel, rho = cuda(np.full(sdf.shape, 1800.0), prec), cuda(np.full(sdf.shape, 1000.0), prec)
    a, b = _last_sample(lambda wv: ib.ib_forward(t, vel, cuda(wv, prec), cuda(src), cuda(rec), dt, 50, rho=rho),
                        inputs.ricker(60.0, dt, 50, t0=0.0), float("inf"))
    assert np.abs(a[:, -1]).max() > 0
    assert np.isfinite(b).all() and np.array_equal(a, b)


@pytest.mark.parametrize("prec", [torch.float32, torch.float64])
@pytest.mark.parametrize("ndim", [2, 3])
def test_negative_density(ndim, prec):
    """The pressure does not depend on the sign of a constant density: both coefficients change sign."""
    h = 10.0
    if ndim == 2:
        sdf = inputs.flat_surface_sdf((133, 71), h, 10.3 * h)
        src, rec = np.array([[60.5 * h, 31.5 * h]]), np.array([[x * h, 12 * h] for x in range(3, 130, 4)])
    else:
        sdf, zs = small_hills()
        src = np.array([[20 * h, 17 * h, 26 * h]])
        rec = np.array([[x * h, y * h, zs[y, x] + 2 * h] for x in range(4, 36, 5) for y in range(4, 32, 5)])
    dt = 0.3 * h / 1800.0
    t = ib.ib_build_stencils(cuda(sdf), h, "free", "staggered", 4)
    wv = inputs.ricker(60.0, dt, 50, t0=0.0)
    a, b = [ib.ib_forward(t, cuda(np.full(sdf.shape, 1800.0), prec), cuda(wv, prec), cuda(src), cuda(rec), dt, 50,
                          rho=cuda(np.full(sdf.shape, r), prec)).double().cpu().numpy() for r in (1000.0, -1000.0)]
    ib.ib_sync_status()
    assert np.abs(a[:, -1]).max() > 0
    assert np.array_equal(a, b)      # every product changes sign and nothing else
