"""The tree build at the edges of its 1024-particle tiles: sets that end at,
before and after a tile, clumps and runs of coincident particles that straddle
one, far fewer particles than the context holds (tiles without any), and every
bucket and group bound at the ends of its range.  Node and group counts, each
group's first particle and size, and the listed pairs equal the definition's
exactly."""
import numpy as np
import pytest

import oracle as O
from test_gpu_tree import morton_sorted, top_down

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("bucket,group", [(1, 1), (1, 64), (7, 8), (8, 32), (14, 14), (14, 64)])
@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 2112, 5000])
def test_tree_tiles(dzs, n, bucket, group):
    rng = np.random.default_rng(n)
    u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64)
    if n > 1000:  # clumps of 200 particles and 30 coincident ones in Morton order about the tile ends
        us, _ = morton_sorted(u.astype(np.uint32))
        u = us.astype(np.uint64)
        u[:, 920:1010] = u[:, 920:921] + rng.integers(0, 2 ** 12, size=(3, 90), dtype=np.uint64)
        u[:, 1010:min(n, 1040)] = u[:, 1010:1011]
    us, keys = morton_sorted((u % 2 ** 32).astype(np.uint32))
    kw = dict(n1d=32, mesh=32, box=64.0, leaf_bucket=bucket, walk_group=group)
    P = O.params(**kw)
    nodes, groups = top_down(keys, bucket, group)
    st, ct = O.groups(P, us)
    k = np.ones(n, np.uint32)
    state = dict(u=us, p=np.zeros((3, n)), g=np.zeros((3, n)), k=k, id=np.arange(n, dtype=np.uint32),
                 fl=np.zeros(n, np.uint8))
    with dzs.Context(**kw, precision=1) as ctx:
        ctx.set_state(state, 0)
        ctx.accel()
        cnt = ctx.counters()
        first, count, _ = ctx.walk_lists()
    assert cnt[3] == 0 and (cnt[0], cnt[1]) == (groups, nodes)
    assert np.array_equal(first, st) and np.array_equal(count, ct)
    assert cnt[2] == O.interaction_count(P, us, k)
