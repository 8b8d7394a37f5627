"""FP64 short-range force where the pair table ends, against the oracle: pairs
closer than the table's smallest z (tiny softening), a cut beyond its largest,
softened pairs, merged multiplicities.  Tolerance of the FP64 force parity:
1e-9 of |g| + 1e-3 g_rms."""
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


@pytest.mark.parametrize("soft,rcut", [(1.0 / 40.0, 4.5), (1e-6, 4.5), (1.0 / 40.0, 6.5), (0.3, 3.0), (1e-6, 6.5)])
@pytest.mark.parametrize("walk_eval", [1, 2])
def test_fp64_walk_table_edges(dzs, soft, rcut, walk_eval):
    kw = dict(n1d=16, mesh=32, box=32.0, merge_level=2, soft_frac=soft, rcut_rs=rcut)
    rng = np.random.default_rng(int(1e6 * soft) + int(10 * rcut))
    n = 4096
    u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64)
    close = rng.integers(0, n, size=n // 3)  # partners at log-uniform separations down to a few lattice units
    sep = np.exp(rng.uniform(np.log(2.0), np.log(2.0 ** 28), (3, n // 3)))
    u[:, :n // 3] = u[:, close] + np.round(sep).astype(np.uint64)
    u = (u % 2 ** 32).astype(np.uint32)
    k = np.where(rng.random(n) < 0.1, rng.integers(1, 500, size=n), 1).astype(np.uint32)
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=k, id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    want = O.accel(O.params(**kw), u, k)
    with dzs.Context(**kw, precision=1, walk_eval=walk_eval) as ctx:
        ctx.set_state(st, 0)
        got = ctx.accel()
    err, ref = np.linalg.norm(got - want, axis=0), np.linalg.norm(want, axis=0)
    rms = np.sqrt((ref ** 2).mean())
    assert np.all(err <= 1e-9 * (ref + 1e-3 * rms)), float((err / (ref + 1e-3 * rms)).max())
