"""Sweeps with the lattices resident in shared memory (the automatic variant of L = 64 .. 512) against
the half-sweep kernels: every size class and exchange (cluster, grid, rows of whole and of split
uint4), replica counts around a launch's capacity, calls below, at and above the length from which the
resident sweep runs, both cycles, every rule.  Spins are compared bit for bit."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ising():
    from paper_2305_12161_gb300 import ising as m
    m.lib()
    return m


def _same(ising, L, R, calls, t0=0, seed=5, **kw):
    with ising.Ising(L, replicas=R, seed=seed, **kw) as a, \
            ising.Ising(L, replicas=R, seed=seed, variant=ising.VARIANT_WORD, **kw) as b:
        a.t = t0
        b.t = t0
        for n in calls:
            a.sweep(n)
            b.sweep(n)
            for r in sorted({0, 1 % R, R // 2, R - 1}):
                assert np.array_equal(a.get_packed(r), b.get_packed(r)), (L, R, n, r)
        assert a.t == b.t


@pytest.mark.parametrize("cycle", [0, 1])
@pytest.mark.parametrize("L,R", [(64, 1), (64, 19), (64, 39), (64, 160), (64, 320), (128, 1), (128, 19), (128, 20),
                                 (128, 80), (192, 1), (192, 13), (256, 1), (256, 2), (256, 9), (256, 10), (320, 1),
                                 (320, 4), (384, 2), (448, 1), (512, 1), (512, 2)])
def test_equals_the_half_sweep_kernel(ising, L, R, cycle):
    _same(ising, L, R, [1, 2, 3, 12, 13], cycle=cycle)


@pytest.mark.parametrize("rule", [1, 2])
@pytest.mark.parametrize("L", [64, 128, 192, 256, 512])
def test_other_rules(ising, L, rule):
    _same(ising, L, 2, [13, 12], tie=rule)


def test_counter_near_its_end_and_long_calls(ising):
    _same(ising, 64, 3, [40], t0=2**32 - 1 - 40, seed=2**64 - 2)
    _same(ising, 64, 2, [5000])
    _same(ising, 256, 2, [4100])


@pytest.mark.parametrize("L,n", [(64, 17), (192, 6)])
def test_equals_the_oracle(ising, L, n):
    want = oracle.init(L, 7, 0)
    oracle.sweeps(want, 0, n, 7)
    with ising.Ising(L, replicas=1, seed=7) as q:
        q.sweep(n)
        assert np.array_equal(q.get_spins(0), want)


def test_contexts_on_several_streams(ising):
    import torch
    spec = [(256, 3, 1), (512, 1, 2), (320, 2, 3), (64, 5, 4), (256, 1, 5)]
    ctx = [ising.Ising(L, replicas=R, seed=s, stream=torch.cuda.Stream()) for L, R, s in spec]
    for _ in range(20):
        for q in ctx:
            q.sweep(16)
    for (L, R, s), q in zip(spec, ctx):
        q.sync()
        with ising.Ising(L, replicas=R, seed=s) as p:
            p.sweep(320)
            for r in range(R):
                assert np.array_equal(p.get_packed(r), q.get_packed(r)), (L, r)
        q.destroy()


@pytest.mark.parametrize("L", [64, 256])
def test_captured_sweep_replays(ising, L):
    import torch
    stream = torch.cuda.Stream()
    with ising.Ising(L, replicas=2, seed=9, stream=stream) as q, ising.Ising(L, replicas=2, seed=9) as p:
        q.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            q.sweep(12)
        for _ in range(2):  # the graph repeats the draws of t = 0 .. 11
            with torch.cuda.stream(stream):
                g.replay()
            p.t = 0
            p.sweep(12)
        for r in range(2):
            assert np.array_equal(p.get_packed(r), q.get_packed(r))


def test_batches_replayed_on_two_streams(ising):
    # captured cooperative launches of two batches, replayed with nothing waiting between them
    import torch
    specs = [[(256, 3, 1), (512, 1, 9), (64, 4, 20)], [(256, 9, 30), (320, 1, 50)]]
    times = [12, 40, 41, 80]
    want = []
    for classes in specs:
        with ising.Batch(classes) as b:
            want.append(b.run(times)[0])
    batches = [ising.Batch(classes, stream=torch.cuda.Stream()) for classes in specs]
    recs = [torch.empty((len(times), b.record_words), dtype=torch.int64, device="cuda") for b in batches]
    torch.cuda.synchronize()
    for _ in range(6):
        for b, rec in zip(batches, recs):
            b.reinit()
            b.run(times, rec=rec, device=True)
    for b, rec, w in zip(batches, recs, want):
        b.sync()
        assert np.array_equal(rec.cpu().numpy(), w)
        b.destroy()


def test_threads_with_different_plans(ising):
    # 135 and 20 KB of shared memory per CTA of one kernel, launched from two threads
    import threading
    import torch
    spec, bad = [(128, 64, 1000 * i + 1) if i % 2 else (128, 12, 1000 * i + 1) for i in range(8)], []
    ctx = [ising.Ising(L, replicas=R, seed=s, stream=torch.cuda.Stream()) for L, R, s in spec]

    def work(q):
        try:
            for _ in range(1500):
                q.sweep(1)
            q.sync()
        except ising.IsingError as e:
            bad.append(str(e))

    threads = [threading.Thread(target=work, args=(q,)) for q in ctx]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for (L, R, s), q in zip(spec, ctx):
        with ising.Ising(L, replicas=1, seed=s + R - 1, variant=ising.VARIANT_WORD) as p:
            p.sweep(1500)
            assert np.array_equal(p.get_packed(0), q.get_packed(R - 1))
        q.destroy()


def _batch_states(b, classes):
    return [b.get_packed(ci, r) for ci, (L, R, _) in enumerate(classes) for r in range(R)]


def _word_states(ising, classes, n):
    """The same sweeps by the one-word-per-thread half-sweep kernel, in a context per class."""
    out = []
    for L, R, seed in classes:
        with ising.Ising(L, replicas=R, seed=seed, variant=ising.VARIANT_WORD) as q:
            q.sweep(n)
            out += [q.get_packed(r) for r in range(R)]
    return out


@pytest.mark.parametrize("classes,launches,without", [
    ([(64, 1, 5), (64, 3, 70), (128, 1, 90), (64, 1, 2**64 - 1), (128, 2, 300)], 2, None),
    # ten 256^3 take three launches, nine (more planes per CTA) one
    ([(192, 1, 1), (256, 1, 20), (192, 2, 30), (256, 2, 40), (512, 1, 50), (256, 7, 60)], 5, 3),
    ([(320, 1, 1), (384, 1, 2), (448, 1, 3), (320, 1, 4)], 3, None)])
def test_batch_classes_of_one_size_share_launches(ising, classes, launches, without):
    n = 24
    want = _word_states(ising, classes, n)
    with ising.Batch(classes) as b:
        l0 = b.launch_count()
        b.sweep(n)
        # one launch per size and group of lattices that fit the device together
        assert b.launch_count() - l0 == launches
        assert all(np.array_equal(x, y) for x, y in zip(_batch_states(b, classes), want))
        b.reinit()
        rec, _ = b.run([5, n])
        assert all(np.array_equal(x, y) for x, y in zip(_batch_states(b, classes), want))
        # a class with a kernel of its own leaves the others together
        if without:
            b.set_class_config(1, variant=ising.VARIANT_ZFAST, tile_z=8)
            b.reinit()
            l0 = b.launch_count()
            b.sweep(n)
            assert b.launch_count() - l0 == without + 2 * n
            assert all(np.array_equal(x, y) for x, y in zip(_batch_states(b, classes), want))


@pytest.mark.parametrize("barrier", [False, True])
@pytest.mark.parametrize("L,R", [(192, 3), (256, 1), (512, 1)])
def test_a_wait_that_runs_out_ends_with_a_status(ising, L, R, barrier):
    # block 0 leaves out a message or a barrier arrival: every block returns, a queued sweep leaves at
    # once, and the context reports the timeout
    import time
    with ising.Ising(L, replicas=R, seed=5) as q:
        q.sweep(16)
        q.sync()
        q.inject_sweep_stall(barrier, timeout_s=0.3)
        t0 = time.time()
        q.sweep(16)
        q.sweep(5000)
        with pytest.raises(ising.IsingError) as e:
            q.sync()
        assert e.value.status == ising.ISING_ETIMEOUT and "resident" in str(e.value)
        assert time.time() - t0 < 10
        with pytest.raises(ising.IsingError) as e:
            q.sweep(1)
        assert e.value.status == ising.ISING_EPOISONED
    _same(ising, L, R, [16])


@pytest.mark.parametrize("read", ["spins", "packed", "radial", "measure"])
def test_a_read_reports_the_timeout(ising, read):
    # the lattice holds messages after a sweep that gave up: no call hands it out as a state
    with ising.Ising(256, replicas=1, seed=5) as q:
        q.inject_sweep_stall(timeout_s=0.3)
        q.sweep(16)
        with pytest.raises(ising.IsingError) as e:
            {"spins": q.get_spins, "packed": q.get_packed, "radial": q.measure_radial, "measure": q.measure}[read]()
        assert e.value.status == ising.ISING_ETIMEOUT


def test_derived_values_of_a_sweep_that_gave_up_are_nan(ising):
    import torch
    with ising.Ising(192, replicas=2, seed=5) as q, ising.Batch([(192, 1, 5)]) as b:
        rec = torch.empty((2, q.record_len), dtype=torch.int64, device="cuda")
        der = torch.zeros((2, 2, 4), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        q.sweep(16)
        q.measure_device(rec, der[0])
        q.inject_sweep_stall(timeout_s=0.3)
        q.sweep(16)
        q.measure_device(rec, der[1])
        torch.cuda.synchronize()
        assert torch.isfinite(der[0, :, :3]).all() and torch.isnan(der[1]).all()
        b.sweep(16)
        assert np.isfinite(b.measure_ex()[1][:, :3]).all()


def test_the_server_reports_the_timeout(ising):
    from paper_2305_12161_gb300 import serve
    srv = serve.QuenchServer(tune=False)
    srv.t0 = 0.0
    srv.submit(serve.Request(id=0, L=192, t_max=16, replicas=1, seed=3, K=1))
    srv._admit()
    srv.active[0].ctx.inject_sweep_stall(timeout_s=0.3)
    with pytest.raises(ising.IsingError) as e:
        while srv.active:
            for a in srv.active:
                srv._issue(a)
            srv._retire()
    assert e.value.status == ising.ISING_ETIMEOUT and not srv.results
