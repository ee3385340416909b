"""Order of launches on a stream and between streams: the option pdl = 0 in the measurement."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    from paper_2305_12161_gb300 import ising as m
    m.lib()
    return m


class _EdgeData(ctypes.Structure):  # cudaGraphEdgeData
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


def _programmatic_edges(stream, enqueue):
    """Programmatic edges of the graph that `enqueue` leaves on `stream` while it is captured."""
    rt = ctypes.CDLL("libcudart.so.13")
    s, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t(0)
    assert rt.cudaStreamBeginCapture(s, 1) == 0  # thread local
    enqueue()
    assert rt.cudaStreamEndCapture(s, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetEdges(graph, None, None, None, ctypes.byref(n)) == 0
    a, b, e = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (_EdgeData * n.value)()
    assert rt.cudaGraphGetEdges(graph, a, b, e, ctypes.byref(n)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return sum(d.type == 1 for d in e)


@pytest.mark.parametrize("L,kw", [(64, {}), (256, {}), (64, {"form": 1}), (512, {}), (16, {})])
def test_measurement_in_plain_stream_order(ising, L, kw):
    import torch
    stream = torch.cuda.Stream()
    edges, recs = {}, {}
    for pdl in (0, 1):
        with ising.Ising(L, replicas=2, seed=3, stream=stream, pdl=pdl, **kw) as q:
            rec = torch.empty((2, q.record_len), dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            q.measure_device(rec)  # allocates the scratch of L = 512
            q.sync()
            recs[pdl] = rec.cpu().numpy()
            edges[pdl] = _programmatic_edges(stream, lambda: (q.measure_device(rec), q.measure_device(rec)))
    assert edges[0] == 0 and edges[1] > 0
    assert np.array_equal(recs[0], recs[1])
