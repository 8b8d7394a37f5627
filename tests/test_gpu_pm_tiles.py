"""CIC deposit and interpolation tiles against the oracle: one tile that is its
own neighbour (mesh 8), meshes coarser and finer than the particle lattice
(every depth of the shared cell table), dense cells, empty tiles, merged
multiplicities, periodic edges.

Tolerances: FP64 the parity bounds (delta 1e-12 of its largest value, PM
acceleration 1e-9 of |g| + 1e-3 g_rms); FP32 delta: a node adds at most 8 cell
sums of n terms, each rounded, 2^-24 (n_cell + 8) < 1e-4 of the largest value
for the 1000 members of the densest cells; PM acceleration 99.9th percentile
1e-4."""
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


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n1d,mesh", [(16, 8), (64, 16), (16, 16), (8, 64), (32, 64), (12, 32), (16, 128)])
def test_pm_tiles(dzs, n1d, mesh, precision):
    kw = dict(n1d=n1d, mesh=mesh, box=float(n1d), merge_level=1)
    rng = np.random.default_rng(n1d * 1000 + mesh)
    n = n1d ** 3 - 7
    u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64)
    clump = n // 4
    side = 2 ** 32 // mesh
    u[:, :clump] = rng.integers(0, mesh, (3, 1 + clump // 1000), dtype=np.uint64)[:, np.arange(clump) // 1000] * np.uint64(side) \
        + rng.integers(0, side, (3, clump), dtype=np.uint64)
    u[0, clump:clump + n // 8] = 2 ** 32 - 1 - u[0, clump:clump + n // 8] % np.uint64(side)  # the periodic face
    u = (u % 2 ** 32).astype(np.uint32)
    k = np.where(rng.random(n) < 0.2, rng.integers(1, 60, size=n), 1).astype(np.uint32)
    st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=k, id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    P = O.params(**kw)
    with dzs.Context(**kw, precision=precision) as ctx:
        ctx.set_state(st, 0)
        got = ctx.accel(dzs.ACC_PM)
        delta = ctx.mesh(dzs.MESH_DELTA)
    wd = O.cic_delta(P, u, k)
    assert np.abs(delta - wd).max() <= (1e-12 if precision else 1e-4) * np.abs(wd).max()
    want = O.accel(P, u, k, parts=1)
    err, ref = np.linalg.norm(got - want, axis=0), np.linalg.norm(want, axis=0)
    rel = err / (ref + 1e-3 * np.sqrt((ref ** 2).mean()))
    assert (rel.max() <= 1e-9) if precision else (np.quantile(rel, 0.999) <= 1e-4), rel.max()
