"""Order of launches on a stream and between streams: the option pdl = 0 in the measurement, and
cooperative launches of contexts and batches on streams of their own."""
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


def test_replayed_batch_waits_for_a_context_s_resident_sweep(ising):
    # 144 CTAs each, more than one per SM together: the replay waits, although CTAs this small could share
    # an SM
    import torch
    times, classes = [4, 8], [(192, 3, 1)]
    with ising.Batch(classes) as b:
        want, _ = b.run(times)
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    with ising.Ising(192, replicas=3, seed=9, stream=sa) as q, ising.Batch(classes, stream=sb) as b:
        rec = torch.empty((len(times), b.record_words), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        q.sweep(16)
        b.run(times, rec=rec, device=True)  # captures
        b.reinit()
        q.sync()
        b.sync()
        ea, eb = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        q.sweep(4000)
        ea.record(sa)
        b.run(times, rec=rec, device=True)
        eb.record(sb)
        q.sync()
        b.sync()
        assert ea.elapsed_time(eb) > 0
        assert np.array_equal(rec.cpu().numpy(), want)


def test_resident_sweeps_that_fit_run_side_by_side(ising):
    # 48 CTAs each: the short call ends inside the long one; two more fill the device and a fourth waits
    import torch
    streams = [torch.cuda.Stream() for _ in range(4)]
    ctx = [ising.Ising(192, replicas=1, seed=40 + i, stream=s) for i, s in enumerate(streams)]
    for q in ctx:
        q.sweep(4)
        q.sync()
    ev = [torch.cuda.Event(enable_timing=True) for _ in ctx]
    for q, s, e, n in zip(ctx, streams, ev, (8000, 8, 8000, 8)):
        q.sweep(n)
        e.record(s)
    for q in ctx:
        q.sync()
    assert ev[1].elapsed_time(ev[0]) > 0
    for i, q in enumerate(ctx):
        with ising.Ising(192, replicas=1, seed=40 + i, variant=ising.VARIANT_WORD) as p:
            p.sweep(q.t)
            assert np.array_equal(p.get_packed(0), q.get_packed(0)), i
        q.destroy()


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_many_contexts_in_any_order(ising, seed):
    # widths from 12 to 150 CTAs on eleven streams, in a random order
    import torch
    rng = np.random.default_rng(seed)
    spec = [(192, 1), (192, 3), (192, 12), (256, 1), (256, 2), (256, 9), (320, 1), (320, 4), (384, 1), (512, 1), (192, 1)]
    ctx = [ising.Ising(L, replicas=R, seed=100 * i + 1, stream=torch.cuda.Stream()) for i, (L, R) in enumerate(spec)]
    for _ in range(120):
        ctx[int(rng.integers(len(ctx)))].sweep(int(rng.integers(3, 40)))
    for (L, R), q, i in zip(spec, ctx, range(len(spec))):
        q.sync()
        with ising.Ising(L, replicas=R, seed=100 * i + 1) as p:
            p.sweep(q.t)
            for r in range(R):
                assert np.array_equal(p.get_packed(r), q.get_packed(r)), (L, R, r)
        q.destroy()


def test_context_sweeps_between_batch_replays(ising):
    import torch
    classes, times = [(512, 1, 9), (256, 2, 30)], [12, 40, 41, 80]
    with ising.Batch(classes) as b:
        want, _ = b.run(times)
    with ising.Ising(512, replicas=1, seed=4) as p, ising.Ising(320, replicas=2, seed=6) as r:
        p.sweep(6 * 24)
        r.sweep(6 * 24)
        states = [p.get_packed(0), r.get_packed(1)]
    with ising.Ising(512, replicas=1, seed=4, stream=torch.cuda.Stream()) as p, \
            ising.Ising(320, replicas=2, seed=6, stream=torch.cuda.Stream()) as r, \
            ising.Batch(classes, stream=torch.cuda.Stream()) as b:
        rec = torch.empty((len(times), b.record_words), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        for _ in range(6):
            p.sweep(24)
            b.reinit()
            b.run(times, rec=rec, device=True)
            r.sweep(24)
        for o in (p, r, b):
            o.sync()
        assert np.array_equal(rec.cpu().numpy(), want)
        assert np.array_equal(p.get_packed(0), states[0]) and np.array_equal(r.get_packed(1), states[1])


def test_batch_sweep_in_a_caller_s_capture(ising):
    # no resident grid there: the classes run on the persistent kernel and as streamed half-sweeps
    import torch
    classes, n = [(192, 2, 3), (256, 2, 8), (64, 2, 50)], 12
    with ising.Batch(classes) as a:
        a.sweep(n)
        want = [a.get_packed(ci, r) for ci, c in enumerate(classes) for r in range(c[1])]
    stream = torch.cuda.Stream()
    with ising.Batch(classes, stream=stream) as b:
        b.sync()
        g = torch.cuda.CUDAGraph()
        l0 = b.launch_count()
        with torch.cuda.graph(g, stream=stream):
            b.sweep(n)
        assert b.launch_count() - l0 == 1 + 2 * n
        with torch.cuda.stream(stream):
            g.replay()
        got = [b.get_packed(ci, r) for ci, c in enumerate(classes) for r in range(c[1])]
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
