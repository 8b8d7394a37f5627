"""The bins of P(k), which a warp adds to from different lanes in successive
rounds of 32 modes: repeated calls agree bit for bit, and the first two bins of a
call with two bins (every round ends in them) equal those of a call with M / 2
bins to the rounding of two orders of summation of positive terms, 64 roundings
of 2^-53 at most."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("mesh", [16, 48, 64, 256])
def test_rows(dzs, mesh, precision):
    if precision and mesh == 256:
        pytest.skip("FP64 meshes are covered by the smaller ones")
    rng = np.random.default_rng(mesh)
    n = 16 ** 3
    st = dict(u=rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32), p=np.zeros((3, n)),
              g=np.zeros((3, n)), k=np.ones(n, np.uint32), id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
    with dzs.Context(n1d=16, mesh=mesh, box=32.0, merge_level=1, precision=precision) as ctx:
        ctx.set_state(st, 0)
        few = ctx.power_spectrum(2, shot=False)
        many = ctx.power_spectrum(mesh // 2, shot=False)
        for _ in range(20):
            for x, y in zip(ctx.power_spectrum(mesh // 2, shot=False), many):
                assert np.array_equal(x, y)
    assert np.array_equal(few[2], many[2][:2])
    assert np.all(np.abs(few[1] - many[1][:2]) <= 64 * 2.0 ** -53 * few[1])
