"""The walk's queue of opened leaves' particles and its COM-first node test: the
listed pairs equal the oracle's interaction count exactly and the FP64 tree
force matches it (1e-9 of the largest), with

  - leaves of 14 that overflow the queue in one round (theta small: every node
    within r_cut is opened), leaves of one particle, and the usual bucket;
  - opening angles on both sides of 1/sqrt(3), above which a node whose cube
    touches the group's may have its COM too far away to be opened by distance."""
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


def particles(name):
    rng = np.random.default_rng(11)
    if name == "cells":  # 14 particles in each of 8^3 cells
        cell = np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij")).reshape(3, -1)
        u = np.repeat(cell, 14, axis=1) * 2 ** 29 + rng.integers(0, 2 ** 29, size=(3, 14 * 512))
    else:
        u = rng.integers(0, 2 ** 32, size=(3, 5003))
    k = np.where(rng.random(u.shape[1]) < 0.2, rng.integers(1, 50, size=u.shape[1]), 1)
    return u.astype(np.uint32), k.astype(np.uint32)


@pytest.mark.parametrize("bucket,group", [(1, 8), (8, 32), (14, 14), (14, 64)])
@pytest.mark.parametrize("theta", [0.05, 0.5, 0.58, 0.9])
@pytest.mark.parametrize("name", ["cells", "uniform"])
def test_lists_and_force(dzs, name, theta, bucket, group):
    kw = dict(n1d=32, mesh=32, box=64.0, theta=theta, leaf_bucket=bucket, walk_group=group)
    P = O.params(**kw)
    u, k = particles(name)
    _, perm = O.sort(u)
    u, k = np.ascontiguousarray(u[:, perm]), k[perm]
    n = u.shape[1]
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=k, id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    want = O.accel(P, u, k, parts=2)
    with dzs.Context(**kw, precision=1) as ctx:
        ctx.set_state(st, 0)
        got = ctx.accel(dzs.ACC_TREE)
        cnt = ctx.counters()
    assert cnt[3] == 0
    assert cnt[2] == O.interaction_count(P, u, k)
    assert np.linalg.norm(got - want, axis=0).max() <= 1e-9 * np.linalg.norm(want, axis=0).max()
