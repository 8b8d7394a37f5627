"""FoF where the cells of friends decide much or nothing against the oracle:
linking lengths from below the finest cell (no cell of friends) to cells of many
particles, coincident particles, dense clumps across cell and box edges.  All
integer work: exact."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

KW = dict(n1d=16, mesh=32, box=32.0, merge_level=2)


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("link", [2e-6, 1.4e-5, 0.01, 0.2, 0.9, 3.5])
@pytest.mark.parametrize("n", [1, 37, 4096])
def test_fof_cells_of_friends(dzs, link, n):
    rng = np.random.default_rng(n)
    u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64)
    # clumps around cell corners (also the box's), with coincident members
    half = n // 2
    corner = rng.integers(0, 8, size=(3, max(1, half // 16))) * 2 ** 29
    c = corner[:, rng.integers(0, corner.shape[1], half)].astype(np.uint64)
    spread = np.exp(rng.uniform(np.log(1.0), np.log(2.0 ** 27), half))
    u[:, :half] = c + np.round(rng.normal(0, 1, (3, half)) * spread).astype(np.int64).astype(np.uint64)
    if half > 8:
        u[:, :4] = u[:, 4:8]
    u = (u % 2 ** 32).astype(np.uint32)
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=rng.integers(1, 9, size=n).astype(np.uint32),
              id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    wh, wlab = O.fof(O.params(**KW), u, st["k"], link=link, nmin=2)
    with dzs.Context(**KW, precision=0) as ctx:
        ctx.set_state(st, 0)
        h, lab = ctx.fof(link=link, nmin=2, labels=True)
    assert np.array_equal(lab, wlab)
    assert len(h) == len(wh)
    for f in ("first", "count", "mass", "rmax2", "x"):
        assert np.array_equal(h[f], wh[f]), f
