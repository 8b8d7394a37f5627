"""The 16-wide FP32 deposit and interpolation tiles (meshes of 2^m, m >= 7, with
fewer than half a particle a cell) at every depth of the shared cell table below
the mesh's: n1d to mesh 1 : 16 (depth raised to the tiles' 8^3 cells) and 1 : 8
(shift 0), 1 : 4 (shift 3), 1 : 2 (shift 6), and the densest set that takes them,
96^3 on mesh 128; tiles that are empty, that hold one clump, and periodic faces.

Tolerances as for the other deposits: delta 2^-24 (n_cell + 8) < 1e-4 of its
largest value for the 1000 members of the densest cells; PM acceleration 99.9th
percentile 1e-4 of |g| + 1e-3 g_rms."""
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


@pytest.mark.parametrize("n1d,mesh", [(8, 128), (16, 128), (32, 128), (64, 128), (96, 128), (64, 256)])
def test_tile_depths(dzs, n1d, mesh):
    assert 2 * n1d ** 3 < mesh ** 3
    kw = dict(n1d=n1d, mesh=mesh, box=float(n1d), merge_level=1)
    rng = np.random.default_rng(n1d + mesh)
    n = n1d ** 3 - 5
    side = 2 ** 32 // mesh
    u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64)
    clump = n // 4
    cells = rng.integers(0, mesh, (3, 1 + clump // 1000), dtype=np.uint64)
    cells[:, :1] = mesh - 1  # the corner cell, whose nodes wrap on every axis
    u[:, :clump] = cells[:, np.arange(clump) // 1000] * np.uint64(side) + rng.integers(0, side, (3, clump), dtype=np.uint64)
    u[1, clump:clump + n // 8] = 2 ** 32 - 1 - u[1, clump:clump + n // 8] % np.uint64(side)  # a periodic face
    u[2, 3 * n // 4:] %= np.uint64(2 ** 30)  # three quarters of the tiles along z hold a third less
    u = u.astype(np.uint32)
    k = np.where(rng.random(n) < 0.2, rng.integers(1, 60, size=n), 1).astype(np.uint32)
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=k, id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    P = O.params(**kw)
    with dzs.Context(**kw) as ctx:
        ctx.set_state(st, 0)
        got = ctx.accel(dzs.ACC_PM)
        delta = ctx.mesh(dzs.MESH_DELTA)
    wd = O.cic_delta(P, u, k)
    assert np.abs(delta - wd).max() <= 1e-4 * np.abs(wd).max()
    want = O.accel(P, u, k, parts=1)
    err, ref = np.linalg.norm(got - want, axis=0), np.linalg.norm(want, axis=0)
    rel = err / (ref + 1e-3 * np.sqrt((ref ** 2).mean()))
    assert np.quantile(rel, 0.999) <= 1e-4, rel.max()
