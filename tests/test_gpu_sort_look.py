"""The radix sort whose waits run out: with no polls allowed, a block that finds
an earlier tile's counts unpublished counts those keys from the pass's input.
Keys and order stay the oracle's, exactly, in the allocation-free call (which
has no status to report a failed wait with) and in a context."""
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
    yield m
    m.dzs_debug_sort_look(-1)


@pytest.mark.parametrize("polls", [0, 1, -1])
@pytest.mark.parametrize("n", [1, 1025, 20011, 100003])
def test_allocation_free_sort(dzs, n, polls):
    import torch
    u = np.random.default_rng(n).integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32)
    u[:, : n // 3] = u[:, n // 3: 2 * (n // 3)]  # ties
    d = torch.from_numpy(u.view(np.int32).copy()).cuda()
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    keys = torch.empty(n, dtype=torch.int64, device="cuda")
    dzs.dzs_debug_sort_look(polls)
    st = dzs.dzs_morton_sort_noalloc(d.data_ptr(), n, perm.data_ptr(), keys.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
    assert st == dzs.DZS_OK
    torch.cuda.synchronize()
    key, want = O.sort(u)
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), want.astype(np.uint32))
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), key[want])


@pytest.mark.parametrize("n", [7169, 60001])
def test_context_sort(dzs, n):
    u = np.random.default_rng(n).integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32)
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=np.ones(n, np.uint32),
              id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    with dzs.Context(n1d=96, mesh=96, box=96.0) as ctx:
        ctx.set_state(st, 0)
        dzs.dzs_debug_sort_look(0)
        ctx.run_stages(dzs.STAGE_SORT)
        got = ctx.state()["id"]
        assert ctx.counters()[3] == 0
    assert np.array_equal(got, O.sort(u)[1].astype(np.uint32))
