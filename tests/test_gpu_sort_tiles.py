"""The radix sort at the edges of its tiles against the oracle's stable Morton
order: sizes around one tile, a single key, several waves of tiles, patterns
whose digits all agree (one counter, one look-back chain) or never do.  The
order is unique, so the comparison is exact."""
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


def positions(rng, n, pattern):
    u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32)
    if pattern == "equal":
        u[:] = u[:, :1]
    elif pattern == "two":
        u = u[:, rng.integers(0, min(2, n), n)]
    elif pattern == "sorted":
        u = u[:, O.sort(u)[1]]
    return np.ascontiguousarray(u)


@pytest.mark.parametrize("pattern", ["random", "equal", "two", "sorted"])
@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 20011, 262143])
def test_small_tiles(dzs, n, pattern):
    import torch
    u = positions(np.random.default_rng(n), n, pattern)
    d = torch.from_numpy(u.view(np.int32).copy()).cuda()
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    keys = torch.empty(n, dtype=torch.int64, device="cuda")
    st = dzs.dzs_morton_sort_noalloc(d.data_ptr(), n, perm.data_ptr(), keys.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    assert st == dzs.DZS_OK
    torch.cuda.synchronize()
    key, want = O.sort(u)
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), want.astype(np.uint32))
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), key[want])


@pytest.mark.parametrize("pattern", ["random", "equal", "sorted"])
@pytest.mark.parametrize("n", [1, 7167, 7168, 7169, 884736])
def test_large_tiles(dzs, n, pattern):
    """a context of 96^3 particle slots takes the large tiles, for any count"""
    u = positions(np.random.default_rng(n + 1), n, pattern)
    st = dict(u=u, p=np.arange(3.0 * n).reshape(3, n), g=np.zeros((3, n)), k=np.ones(n, np.uint32),
              id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    with dzs.Context(n1d=96, mesh=96, box=96.0, precision=1) as ctx:
        ctx.set_state(st, 0)
        ctx.run_stages(dzs.STAGE_SORT)
        s = ctx.state()
    want = O.sort(u)[1]
    assert np.array_equal(s["id"], want.astype(np.uint32))
    assert np.array_equal(s["u"], u[:, want]) and np.array_equal(s["p"], st["p"][:, want])
