"""Steps captured by the caller: the graph's edges are plain ones (launches
overlap only outside a capture), and replaying it advances the state as the
same steps launched directly."""
import ctypes

import pytest
import torch

from gpu_common import dev
from paper_1801_04586_gb300 import Batch, Lattice
from test_gpu_batch import DOMAINS

pytestmark = pytest.mark.gpu

THREAD_LOCAL = 1  # CU_STREAM_CAPTURE_MODE_THREAD_LOCAL


class EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


def driver():
    lib = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        assert getattr(lib, name)(*args) == 0, name
    return call


def capture(stream, work):
    """(graph, dependency types of its edges) of what work() launches on stream."""
    cu, s, graph = driver(), ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    cu("cuStreamBeginCapture_v2", s, THREAD_LOCAL)
    try:
        work()
    finally:
        cu("cuStreamEndCapture", s, ctypes.byref(graph))
    n = ctypes.c_size_t(256)
    a, b, e = (ctypes.c_void_p * 256)(), (ctypes.c_void_p * 256)(), (EdgeData * 256)()
    cu("cuGraphGetEdges_v2", graph, a, b, e, ctypes.byref(n))
    return graph, [e[k].type for k in range(min(n.value, 256))]


def replay(stream, graph):
    cu, s, ex = driver(), ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    cu("cuGraphInstantiateWithFlags", ctypes.byref(ex), graph, ctypes.c_ulonglong(0))
    cu("cuGraphLaunch", ex, s)
    stream.synchronize()
    cu("cuGraphExecDestroy", ex)
    cu("cuGraphDestroy", graph)


@pytest.mark.parametrize("kw", [{}, dict(storage="f16"), dict(storage="f16", wait_cycles=4_000_000_000),
                                dict(pattern="aa"), dict(lattice=27), dict(variant=1)])
def test_captured_steps_have_plain_edges(kw):
    stream = torch.cuda.Stream(dev())
    lats = [Lattice(16, 24, 20, 0.05, walls=4, device=dev(), stream=stream, **kw) for _ in range(2)]
    for g in lats:
        g.set_force_uniform(1e-5)
        g.init_equilibrium()
        g.step(2)  # the first launch of a kernel may set an attribute
    stream.synchronize()
    graph, types = capture(stream, lambda: lats[0].step(6))
    assert len(types) >= 2 and not any(types)
    replay(stream, graph)
    lats[1].step(6)
    stream.synchronize()
    with torch.cuda.stream(stream):
        a, b = (g.populations(deviation=True) for g in lats)
    stream.synchronize()
    assert torch.equal(a, b)
    for g in lats:
        g.close()


@pytest.mark.parametrize("mode", [Batch.DIRECT, Batch.PER_DOMAIN])
def test_captured_batch_steps_have_plain_edges(mode):
    stream = torch.cuda.Stream(dev())
    with torch.cuda.stream(stream):
        bs = [Batch(DOMAINS, device=dev()) for _ in range(2)]
    for b in bs:
        b.init_equilibrium()
        b.step(2, mode)
    stream.synchronize()
    graph, types = capture(stream, lambda: bs[0].step(4, mode))
    assert len(types) >= 3 and not any(types)
    replay(stream, graph)
    bs[1].step(4, mode)
    stream.synchronize()
    with torch.cuda.stream(stream):
        for k in range(len(DOMAINS)):
            assert torch.equal(bs[0].populations(k, deviation=True), bs[1].populations(k, deviation=True))
    for b in bs:
        b.close()
