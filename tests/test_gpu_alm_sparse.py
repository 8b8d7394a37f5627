"""Harmonic analysis of maps with a few occupied pixels against the spherical
harmonics at those pixels' centres: the ring transform with tabulated phasors
(rings of at most 4096 pixels) and without, one and several chunks of rings.

Tolerance: |da_lm| <= 1e-10 Omega sum(map), the bound the definition test uses."""
import math

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("nside,lmax", [(2, 8), (4, 3), (64, 130), (256, 65), (1024, 33), (2048, 70), (4096, 5)])
def test_alm_of_single_pixels(dzs, nside, lmax):
    special = pytest.importorskip("scipy.special")
    rng = np.random.default_rng(nside + lmax)
    npix = 12 * nside * nside
    # the poles, the equator, both belt edges, and random pixels
    pix = np.unique(np.concatenate([[0, npix - 1, npix // 2, 2 * nside * (nside + 1), npix - 2 * nside * (nside + 1) - 1],
                                    rng.integers(0, npix, 40)]))
    v = O.pix2vec(nside, pix)
    rec = np.zeros(len(pix), O.RECORD_DTYPE)
    rec["k"] = rng.integers(1, 1000, size=len(pix))
    rec["a_cross"] = 0.5
    rec["x"] = (16.0 + 8.0 * v).T
    with dzs.Context(n1d=16, mesh=32, box=32.0) as ctx:
        ctx.observe(nside=nside)
        ctx.observe_add_records(rec)
        sky = ctx.skymap(nside)
        cl, a = ctx.skymap_alm(lmax)
    assert np.array_equal(np.flatnonzero(sky), pix)
    theta, phi = np.arccos(v[2]), np.arctan2(v[1], v[0])
    want = np.zeros((lmax + 1, lmax + 1), complex)
    for l in range(lmax + 1):
        for m in range(l + 1):
            want[l, m] = 4 * math.pi / npix * (rec["k"] * np.conj(special.sph_harm_y(l, m, theta, phi))).sum()
    scale = 4 * math.pi / npix * rec["k"].sum()
    assert np.abs(a - want).max() <= 1e-10 * scale
    p = np.abs(want) ** 2
    assert np.allclose(cl, (2 * p.sum(1) - p[:, 0]) / (2 * np.arange(lmax + 1) + 1), rtol=1e-8, atol=1e-18 * scale ** 2)
