"""lambda_mm's factor s^m, s the sine of the colatitude: one pixel on a ring near
the equator against one on the equator, where s = 1.  With m = lmax = the
pixels of a ring the phases are exactly 1 or -1, and the ratio of the two a_mm
is s^m but for roundings: of the power (two words: half a unit and less than a
half more), the leading product, the pixel's value and the ring weight, each side
of the ratio, and the ratio's own comparison in rationals: below 6 units of
2^-53.  (Plain repeated squaring: some tens.)"""
import math
from fractions import Fraction

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


@pytest.mark.parametrize("nside,m", [(64, 256), (32, 128), (128, 512)])
def test_power_of_the_sine(dzs, nside, m):
    assert m == 4 * nside

    def a_mm(ring):
        pix = 2 * nside * (nside - 1) + (ring - nside) * 4 * nside
        rec = np.zeros(1, O.RECORD_DTYPE)
        rec["k"], rec["a_cross"] = 1, 0.5
        rec["x"] = (16.0 + 8.0 * O.pix2vec(nside, np.array([pix]))).T
        with dzs.Context(n1d=16, mesh=32, box=32.0) as ctx:
            ctx.observe(nside=nside)
            ctx.observe_add_records(rec)
            assert np.flatnonzero(ctx.skymap(nside)) == [pix]
            a = ctx.skymap_alm(m)[1][m, m]
        assert a.imag == 0.0
        return Fraction(abs(float(a.real)))

    equator = a_mm(2 * nside)
    off = []
    for j in range(1, nside // 4):
        z = j * 2.0 / (3.0 * nside)
        s = Fraction(math.sqrt((1.0 - z) * (1.0 + z)))
        off.append(float(a_mm(2 * nside - j) / equator / s ** m - 1) * 2.0 ** 53)
    assert max(abs(x) for x in off) <= 6.0, off
