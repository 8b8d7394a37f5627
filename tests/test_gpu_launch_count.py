"""The context's count of launched kernels (dzs_get_counters [4]) against counts
taken from outside the library: a step captured into a CUDA graph, whose kernel
nodes are counted, and the profiler's kernel records for the calls that
synchronise (P(k), FoF, forces, state)."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dzs():
    from paper_2005_05328_gb300 import build
    build.build()
    import paper_2005_05328_gb300 as m
    m.load()
    return m


def captured_kernels(stream, fn):
    cu = ctypes.CDLL("libcuda.so.1")
    s, g, n = ctypes.c_void_p(stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(s, 2) == 0  # relaxed
    fn()
    assert cu.cuStreamEndCapture(s, ctypes.byref(g)) == 0
    assert cu.cuGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    kind, kernels = ctypes.c_int(), 0
    for x in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(x), ctypes.byref(kind)) == 0
        kernels += kind.value == 0
    assert cu.cuGraphDestroy(g) == 0
    return kernels


# record, tile and row-major deposits; both criteria and no merging; FP32 and FP64
@pytest.mark.parametrize("kw", [dict(n1d=16, mesh=32), dict(n1d=16, mesh=32, precision=1), dict(n1d=16, mesh=128),
                                dict(n1d=16, mesh=24), dict(n1d=12, mesh=24, precision=1),
                                dict(n1d=48, mesh=96, dzs_criterion=1), dict(n1d=16, mesh=32, dzs_on=0)])
def test_step(dzs, kw):
    import torch
    stream = torch.cuda.Stream()
    with dzs.Context(**kw, box=32.0, merge_level=1, stream=stream.cuda_stream) as ctx:
        ctx.ics()
        ctx.step(1)
        before = ctx.counters()[4]
        kernels = captured_kernels(stream.cuda_stream, lambda: ctx.step(1))
        assert kernels > 0 and ctx.counters()[4] - before == kernels


@pytest.mark.parametrize("kw", [dict(n1d=16, mesh=32), dict(n1d=16, mesh=128), dict(n1d=16, mesh=24),
                                dict(n1d=16, mesh=24, precision=1)])
def test_synchronous_calls(dzs, kw):
    import torch
    import torch.profiler as tp

    def profiled(fn):
        with tp.profile(activities=[tp.ProfilerActivity.CUDA]) as p:
            fn()
            torch.cuda.synchronize()
        names = [e.name for e in p.events() if str(e.device_type).endswith("CUDA")]
        return sum(not x.lower().startswith("mem") for x in names)

    with dzs.Context(**kw, box=32.0, merge_level=1) as ctx:
        ctx.ics()
        profiled(ctx.accel)
        if profiled(ctx.accel) == 0:
            pytest.skip("the profiler records no kernels here")
        for fn in (ctx.ics, lambda: ctx.step(1), ctx.accel, lambda: ctx.power_spectrum(8),
                   lambda: ctx.fof(0.2, 2), lambda: ctx.fof(0.2, 2, labels=True), ctx.state, ctx.diagnostics):
            before = ctx.counters()[4]
            kernels = profiled(fn)
            assert kernels > 0 or kw.get("precision") == 1
            assert ctx.counters()[4] - before == kernels
