"""The radix sort of a large context (capacity from 2^19 on), whose tiles follow
the count on the device: counts at the edges where a thread takes 2, 6 or 14 keys
(512 threads a block; waves of 152 blocks in a 96^3 context, of 304 in a 192^3
one), from one tile to the largest tiles, against the oracle's stable Morton order,
exactly; and a count that shrinks from call to call in one context, as DZS shrinks
it."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

SLOTS = {96: 152, 192: 304}  # blocks of a wave


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


@pytest.fixture(scope="module", params=[96, 192])
def ctx(dzs, request):
    with dzs.Context(n1d=request.param, mesh=96, box=2.0 * request.param) as c:
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
@pytest.mark.parametrize("keys,plus", [(14, 1), (14, 0), (6, 1), (6, 0), (6, -1), (2, 1), (2, 0), (2, -1), (1, 1)])
def test_counts(dzs, ctx, keys, plus, pattern):
    n1d = ctx.params.n1d
    check(dzs, ctx, min(n1d ** 3, keys * 512 * SLOTS[n1d] + plus), pattern)


@pytest.mark.parametrize("n", [1, 1024, 1025, 3073])
def test_few(dzs, ctx, n):
    check(dzs, ctx, n, "random")


def test_full_capacity(dzs, ctx):
    check(dzs, ctx, ctx.params.n1d ** 3, "random")
