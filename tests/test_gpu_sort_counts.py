"""The radix sort of a large context (capacity from 2^19 on), whose tiles follow
the count on the device: counts at the edges where a thread takes 2, 6 or 14
keys (304 blocks of 512 threads in a wave), from one tile to the largest tiles, against the oracle's stable Morton order, exactly; and a count
that shrinks from call to call in one context, as DZS shrinks it."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

WAVE = 2 * 152 * 512


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


@pytest.fixture(scope="module")
def ctx(dzs):
    with dzs.Context(n1d=192, mesh=96, box=192.0) as c:  # 7.1M slots
        yield c


def check(dzs, ctx, n, pattern):
    u = np.random.default_rng(n).integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32)
    if pattern == "ties":
        u[:, n // 2:] = u[:, : n - n // 2]
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=np.ones(n, np.uint32),
              id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    ctx.set_state(st, 0)
    ctx.run_stages(dzs.STAGE_SORT)
    assert np.array_equal(ctx.state()["id"], O.sort(u)[1].astype(np.uint32))


@pytest.mark.parametrize("pattern", ["random", "ties"])
@pytest.mark.parametrize("n", [14 * WAVE + 1, 14 * WAVE, 6 * WAVE + 1, 6 * WAVE, 6 * WAVE - 1, 2 * WAVE + 1, 2 * WAVE,
                               2 * WAVE - 1, WAVE + 1, 1025, 1024, 1])
def test_counts(dzs, ctx, n, pattern):
    check(dzs, ctx, n, pattern)


def test_full_capacity(dzs, ctx):
    check(dzs, ctx, 192 ** 3, "random")
