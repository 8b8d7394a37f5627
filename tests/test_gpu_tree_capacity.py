"""A set whose oct-tree outgrows the node capacity (2 cap + 1024): no block may
write a node, whichever lane of its first warp sees that there is no tree.  The
call reports DZS_EOVERFLOW, the tree is empty, and the next state is served.

Close pairs, leaves of one particle: a pair splits at depth 20, so that each
owns a chain of nodes, 16 particle slots in all needing more than four times
the capacity.  One to four tiles of 1024 particles."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

KW = dict(n1d=16, mesh=32, box=32.0, merge_level=1, leaf_bucket=1, walk_group=8)


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


def state(u):
    n = u.shape[1]
    return dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=np.ones(n, np.uint32),
                id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))


@pytest.mark.parametrize("n", [1024, 2050, 4096])
def test_tree_over_capacity_writes_nothing(dzs, n):
    rng = np.random.default_rng(n)
    pairs = n // 2
    first = rng.integers(0, 2 ** 32, size=(3, pairs), dtype=np.uint64).astype(np.uint32)
    second = first.copy()
    second[0] ^= np.uint32(1 << 12)  # the two part at depth 20
    u = np.concatenate([first, second], axis=1)
    capacity = n  # of particles: the node capacity follows it
    assert pairs * (20 - 5) > 2 * capacity + 1024  # at depth 5 (32768 cells) nearly every pair is alone
    with dzs.Context(**KW, capacity=capacity, precision=1) as ctx:
        ctx.set_state(state(u), 0)
        with pytest.raises(dzs.DzsError) as e:
            ctx.accel()
        assert e.value.status == dzs.DZS_EOVERFLOW
        cnt = ctx.counters()
        assert cnt[0] == 0 and cnt[1] == 0 and cnt[3] & 1, cnt
        # an ordinary set afterwards
        v = rng.integers(0, 2 ** 32, size=(3, n // 2), dtype=np.uint64).astype(np.uint32)
        ctx.set_state(state(v), 0)
        got = ctx.accel()
        assert ctx.counters()[3] == 0
    want = O.accel(O.params(**KW), v, np.ones(n // 2, np.uint32))
    err, ref = np.linalg.norm(got - want, axis=0), np.linalg.norm(want, axis=0)
    assert np.all(err <= 1e-9 * (ref + 1e-3 * np.sqrt((ref ** 2).mean())))
