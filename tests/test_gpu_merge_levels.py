"""The merge where levels are skipped by distance, against the oracle's
recursion: every opening angle from deep to none, cell sizes from one lattice
spacing to the largest, lightcones inside and outside the set, both criteria,
cells above the direct-sum size; and several merges in a row on one context.
Integers and the FP64 momentum sums are compared exactly."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

TWO32 = 2 ** 32


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


def clustered(seed, n):
    rng = np.random.default_rng(seed)
    u = rng.integers(0, TWO32, size=(3, n), dtype=np.uint64)
    c = rng.integers(0, TWO32, size=(3, 12), dtype=np.uint64)
    half = n // 2
    which = rng.integers(0, 12, half)
    spread = (2.0 ** rng.uniform(18, 29, 12))[which]
    u[:, :half] = c[:, which] + np.round(np.abs(rng.normal(0, 1, (3, half))) * spread).astype(np.uint64)
    u = (u % TWO32).astype(np.uint32)
    u = np.ascontiguousarray(u[:, O.sort(u)[1]])
    return dict(u=u, p=rng.normal(0, 1, (3, n)), g=rng.normal(0, 1, (3, n)) * 10.0 ** rng.uniform(-3, 1, n),
                k=rng.integers(1, 9, size=n).astype(np.uint32), id=rng.permutation(n).astype(np.uint32),
                fl=rng.integers(0, 2, n).astype(np.uint8))


@pytest.mark.parametrize("criterion", [0, 1])
@pytest.mark.parametrize("level", [1, 3, 5])
@pytest.mark.parametrize("theta", [0.03, 0.1, 0.5, 0.9])
def test_merge_levels(dzs, theta, level, criterion):
    kw = dict(n1d=16, mesh=32, box=32.0, merge_level=level, theta_dzs=theta, alpha_dyn=0.3)
    P = O.params(**kw, criterion=criterion)
    with dzs.Context(**kw, dzs_criterion=criterion, precision=1) as ctx:
        for seed, frac in ((1, 0.0), (2, 0.1), (3, 0.35), (4, 0.6), (5, 0.95)):
            st = clustered(seed, 4096 - 11 * seed)
            want = O.merge(P, int(frac * TWO32), st)
            ctx.set_state(st, 10)
            ctx.merge_only(int(frac * TWO32))
            got = ctx.state()
            for name in ("u", "k", "id", "fl", "p"):
                assert np.array_equal(got[name], want[name]), (frac, name)
