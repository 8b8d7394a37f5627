"""The FP64 sums of P(k) in an FP32 context.  All particles sit on one mesh node,
one cell from the corner along x, so that the deposit and every butterfly of the
mesh 16 transform are exact and |delta_k|^2 = M^6 (c^2 + s^2) with c, s the FP32
cosine and sine of 2 pi kx / 16: the square needs 48 bits, its sum more.  P(k) is
then known but for the FP64 roundings of weights and sums: some 6 a mode and at
most 24 along a sum of positive terms, at random 0.29 sqrt(30) = 1.6 units of
2^-53, five times that allowed.  (Squares summed in two FP32 words stay 5 to 30
units low: their errors are alike in every mode.)"""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

M, N1D, BOX = 16, 8, 16.0


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


def expected(nbins):
    f32 = np.float32
    e = [Fraction(float(f32(math.cos(2 * math.pi * k / M)))) ** 2 + Fraction(float(f32(math.sin(2 * math.pi * k / M)))) ** 2
         for k in range(M)]
    # the per-axis CIC window as the context tabulates it
    w = []
    for k in range(M):
        m = k if k <= M // 2 else k - M
        x = math.pi * m / M
        s = math.sin(x) / x if m else 1.0
        w.append(Fraction(float(f32(s * s))))
    tot, cnt = [Fraction(0)] * (nbins + 1), [0] * (nbins + 1)
    signed = [k if k <= M // 2 else k - M for k in range(M)]
    for kx in range(M):
        for ky in range(M):
            for kz in range(M):
                n2 = signed[kx] ** 2 + signed[ky] ** 2 + signed[kz] ** 2
                b = 0
                while not (b * b - b < n2 <= b * b + b) and n2 > 0:
                    b += 1
                if 1 <= b <= nbins:
                    # (kx and -kx have the same table entries up to sign)
                    tot[b] += e[min(kx, M - kx)] / (w[kx] * w[ky] * w[kz]) ** 2
                    cnt[b] += 1
    return [tot[b] / cnt[b] * Fraction(BOX) ** 3 for b in range(1, nbins + 1)], cnt[1:]


def test_fp32_context_sums_in_fp64(dzs):
    n = N1D ** 3
    u = np.zeros((3, n), np.uint32)
    u[0] = 2 ** 32 // M
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=np.ones(n, np.uint32),
              id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    with dzs.Context(n1d=N1D, mesh=M, box=BOX, merge_level=1) as ctx:
        ctx.set_state(st, 0)
        _, pk, nm = ctx.power_spectrum(M // 2, shot=False)
    want, cnt = expected(M // 2)
    assert np.array_equal(nm, cnt)
    off = [float((Fraction(float(p)) - q) / q) * 2.0 ** 53 for p, q in zip(pk, want)]
    assert max(abs(x) for x in off) <= 8.0, off
