"""FP32 short-range force on the paired instructions against the oracle: lists
of odd and even length, a single group, self pairs, softened pairs, merged
multiplicities, and a cut beyond the fitted polynomial's range (formula path).

Tolerance (the library's FP32 bound): the 99.9th percentile of |dg| / (|g| +
1e-3 g_rms) at most 1e-4.  Two particles at an offset of FP32 rounding
(2^-24 of the group's reach) lose more, so the largest may reach 1e-2."""
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


@pytest.mark.parametrize("soft,rcut", [(1.0 / 40.0, 4.5), (0.3, 4.5), (1.0 / 40.0, 6.5), (0.3, 2.0)])
@pytest.mark.parametrize("n", [1, 2, 3, 9, 33, 100, 4095])
def test_fp32_walk(dzs, soft, rcut, n):
    kw = dict(n1d=16, mesh=32, box=32.0, merge_level=2, soft_frac=soft, rcut_rs=rcut)
    rng = np.random.default_rng(n + int(10 * rcut))
    u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64)
    if n < 500:  # few particles: close enough to interact
        u = 2 ** 31 + u // 32
    k = np.where(rng.random(n) < 0.2, rng.integers(1, 50, size=n), 1).astype(np.uint32)
    u = u.astype(np.uint32)
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=k, id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    want = O.accel(O.params(**kw), u, k, parts=2)  # the tree part: exactly zero for one particle
    with dzs.Context(**kw, precision=0) as ctx:
        ctx.set_state(st, 0)
        got = ctx.accel(dzs.ACC_TREE)
        again = ctx.accel(dzs.ACC_TREE)
    assert np.array_equal(got, again)
    err, ref = np.linalg.norm(got - want, axis=0), np.linalg.norm(want, axis=0)
    rel = err / (ref + 1e-3 * np.sqrt((ref ** 2).mean()) + 1e-300)
    assert np.quantile(rel, 0.999 if n > 1000 else 0.9) <= 1e-4 and rel.max() <= 1e-2, rel.max()
