"""The PM Poisson solve at every transform length of the library, against an
FP64 FFT of the density the library deposited.

Tolerance: a length-n FP32 FFT has a relative rms error of about
eps sqrt(log2 n) with eps = 2^-24; two 3D transforms (6 passes of log2 n <= 9
stages) and the Green factor (three rounded tables, one division) stay below
eps (sqrt(6 * 9) + 5) < 8e-7 in the 2-norm, and 6 standard deviations of that
per mesh point.  FP64: the same with eps = 2^-53."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


def phi_of(delta, box, rs, omega_m):
    m = delta.shape[0]
    kf = 2.0 * math.pi / box
    n = np.fft.fftfreq(m, 1.0 / m)
    h = np.arange(m // 2 + 1)
    k2 = kf * kf * (n[:, None, None] ** 2 + n[None, :, None] ** 2 + h[None, None, :] ** 2)
    w = (np.sinc(n / m) ** 2)[:, None, None] * (np.sinc(n / m) ** 2)[None, :, None] * (np.sinc(h / m) ** 2)[None, None]
    k2[0, 0, 0] = 1.0
    g = -1.5 * omega_m * np.exp(-k2 * rs * rs) / (k2 * w * w)
    g[0, 0, 0] = 0.0
    return np.fft.irfftn(np.fft.rfftn(delta) * g, s=delta.shape, axes=(0, 1, 2))


@pytest.mark.parametrize("precision,mesh", [(0, m) for m in (8, 16, 24, 32, 64, 96, 128, 192, 256, 384, 512)]
                         + [(1, m) for m in (8, 12 * 2, 32, 64, 96, 128, 256)])
def test_potential_matches_fp64_fft(dzs, precision, mesh):
    n1d, box = 16, 32.0
    rng = np.random.default_rng(mesh)
    n = n1d ** 3
    st = dict(u=rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32), p=np.zeros((3, n)),
              g=np.zeros((3, n)), k=np.ones(n, np.uint32), id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    with dzs.Context(n1d=n1d, mesh=mesh, box=box, precision=precision, dzs_on=0) as ctx:
        ctx.set_state(st, 0)
        ctx.accel(dzs.ACC_PM)
        delta, phi = ctx.mesh(dzs.MESH_DELTA), ctx.mesh(dzs.MESH_PHI)
        p = ctx.params
        want = phi_of(delta, box, p.rs_cells * box / mesh, p.omega_m)
    rms = math.sqrt((want ** 2).mean())
    err = np.abs(phi - want)
    tol = 8e-7 if precision == 0 else 8e-7 * 2.0 ** -29
    assert math.sqrt((err ** 2).mean()) <= tol * rms
    assert err.max() <= 6 * tol * max(rms, np.abs(want).max())


@pytest.mark.parametrize("mesh,nbins", [(8, 1), (8, 4), (16, 7), (24, 12), (32, 16), (96, 41), (256, 128)])
def test_power_spectrum_bins(dzs, mesh, nbins):
    """Counts exact, mean |k| to FP64 rounding, P(k) of a random set against
    numpy sums over the same modes (FP64 contexts: 1e-12 of the bin's power;
    the small meshes cover one split per plane and rows shorter than a warp)"""
    n1d, box = 16, 32.0
    rng = np.random.default_rng(mesh + nbins)
    n = n1d ** 3
    st = dict(u=rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32), p=np.zeros((3, n)),
              g=np.zeros((3, n)), k=np.ones(n, np.uint32), id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    with dzs.Context(n1d=n1d, mesh=mesh, box=box, precision=1, dzs_on=0) as ctx:
        ctx.set_state(st, 0)
        k, pk, modes = ctx.power_spectrum(nbins, shot=False)
        delta = ctx.mesh(dzs.MESH_DELTA)
    f = np.fft.fftfreq(mesh, 1.0 / mesh)
    n2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2
    w = np.sinc(f / mesh) ** 2
    power = np.abs(np.fft.fftn(delta)) ** 2 * (box / mesh ** 2) ** 3 / (
        w[:, None, None] * w[None, :, None] * w[None, None, :]) ** 2
    b = np.floor(np.sqrt(n2) + 0.5).astype(int)
    for q in range(1, nbins + 1):
        sel = b == q
        assert modes[q - 1] == sel.sum()
        assert k[q - 1] == pytest.approx(2 * math.pi / box * np.sqrt(n2[sel]).mean(), rel=1e-13)
        assert pk[q - 1] == pytest.approx(power[sel].mean(), rel=1e-12)
