"""Calls beside other work: two host threads, a busy GPU, a caller's stream of
another priority or on a part of the GPU. Counts are compared with the ones the
same calls give alone."""
import threading
import time

import numpy as np
import pytest

import graphgen
import paper_1608_05138_gb300 as gcb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1608_05138_gb300 import build
    build.build()


def run_threads(*targets):
    """Runs them side by side; the first exception is raised here."""
    errors = []

    def guarded(f):
        try:
            f()
        except BaseException as e:  # noqa: B902
            errors.append(e)

    threads = [threading.Thread(target=guarded, args=(f,)) for f in targets]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_threads_count_dense_graphs_of_different_sizes():
    # dense graphs share a kernel whose shared memory grows with the graph: one
    # thread's count must not narrow what another one launches with
    import torch
    end = time.time() + 6

    def counting(g, x):
        def f():
            while time.time() < end:
                assert g.count() == x
        return f

    handles = [gcb.Graph(*graphgen.er(n, p, n), stream=torch.cuda.Stream()) for n, p in ((64, 0.4), (300, 0.9)) * 8]
    try:
        run_threads(*[counting(g, g.count()) for g in handles])
    finally:
        for g in handles:
            g.close()


def batch_count(g):
    with gcb.Graph(*g) as h:
        return h.count()


def test_batch_goes_on_while_a_thread_captures():
    # the dispatcher queries events and allocates while the caller has a capture
    # of the default mode under way, and the caller submits and polls: neither the
    # capture nor a launch in flight may suffer
    import torch
    large = [graphgen.chung_lu(60000, 500000 + 20000 * i, 2.2, 1e6, 3000.0, 3 + i) for i in range(4)]
    small = [graphgen.er(300 + i, 0.1, i) for i in range(6)]  # of other sizes: buffers grow meanwhile
    expect = [batch_count(g) for g in large + small]
    x = torch.zeros(8, device="cuda")
    b = gcb.gc_batch_create(16 << 30, 0)
    try:
        tickets = [gcb.gc_batch_submit(b, *g) for g in large[:2]]
        for k in range(2):
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                x += 1
                tickets += [gcb.gc_batch_submit(b, *g) for g in [large[2 + k]] + small[3 * k:3 * k + 3]]
                gcb.gc_batch_flush(b)
                time.sleep(0.02)
                last = gcb.gc_batch_poll(b, tickets.pop(), timeout_us=60_000_000)
            assert last == expect[4 + 3 * k + 2]
            graph.replay()
        torch.cuda.synchronize()
        order = [0, 1, 2, 4, 5, 3, 7, 8]
        res = [gcb.gc_batch_poll(b, t, timeout_us=60_000_000) for t in tickets]
    finally:
        gcb.gc_batch_destroy(b)
    assert x.tolist() == [2.0] * 8
    assert res == [expect[i] for i in order]


def test_refused_submissions_take_no_device_memory():
    # a submission that does not fit in the budget now is refused before it is
    # copied and checked on the device; an invalid one gets its own code
    import torch
    rp, ci = graphgen.er(100000, 4e-4, 5)  # 4M entries: 16 MB of CSR
    bad = ci.copy()
    x = int(np.flatnonzero(np.diff(rp) >= 3)[0])
    bad[rp[x]] = bad[rp[x] + 1]
    need = 44 * 100000 + 32 * (len(ci) // 2) + 1024 + 2 * 152 * 100000 * 4
    gcb.gc_release_cached_memory()
    b = gcb.gc_batch_create(need + 10000, gcb.GC_BATCH_MANUAL)
    try:
        t = gcb.gc_batch_submit(b, *graphgen.er(100, 0.5, 1))  # 80 KB of the budget, held until it is launched
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for _ in range(2):
            assert gcb.gc_batch_try_submit(b, rp, ci) is None
        with pytest.raises(gcb.GcError) as ei:
            gcb.gc_batch_submit(b, rp, bad)
        assert ei.value.status == -3
        assert free - torch.cuda.mem_get_info()[0] < 8 << 20
        gcb.gc_batch_flush(b)
        assert gcb.gc_batch_poll(b, t) is not None
        for _ in range(3):  # a refusal gives its share back
            with pytest.raises(gcb.GcError) as ei:
                gcb.gc_batch_submit(b, rp, bad)
            assert ei.value.status == -3
        t = gcb.gc_batch_submit(b, rp, ci)
        gcb.gc_batch_flush(b)
        assert gcb.gc_batch_poll(b, t)[0] == len(ci) // 2
    finally:
        gcb.gc_batch_destroy(b)


@pytest.fixture(scope="module")
def hold_gpu():
    """hold(seconds): kernels whose long-lived CTAs take every thread of the GPU, on the current stream."""
    import torch
    code = "template <typename T> T hold(T x, float n) { for (int i = 0; i < (int)n; ++i) x = x * 1.0000001f + 1e-7f; return x; }"
    fn = torch.cuda.jiterator._create_jit_fn(code, n=1.0)
    x = torch.zeros(torch.cuda.get_device_properties(0).multi_processor_count * 16 * 512 * 4, device="cuda")

    def took(n):
        torch.cuda.synchronize()
        t = time.perf_counter()
        fn(x, n=n)
        torch.cuda.synchronize()
        return time.perf_counter() - t

    took(1e3)
    per = (took(4e5) - took(1e5)) / 3e5
    return lambda seconds: fn(x, n=float(int(seconds / per)))


def test_submitting_does_not_wait_for_running_kernels(hold_gpu):
    # graphs of 2^16 entries or more are checked on the device where it has room
    import torch
    g = graphgen.er(3000, 0.03, 9)
    assert len(g[1]) >= 1 << 16
    bad = g[1].copy()
    bad[g[0][5]] = bad[g[0][5] + 1]
    expect = batch_count(g)
    b = gcb.gc_batch_create(8 << 30, gcb.GC_BATCH_MANUAL)
    try:
        tickets = [gcb.gc_batch_submit(b, *g) for _ in range(8)]  # the blocks and streams exist from here on
        gcb.gc_batch_flush(b)
        assert all(gcb.gc_batch_poll(b, t) == expect for t in tickets)
        hold_gpu(2.0)
        done = torch.cuda.Event()
        done.record()
        worst, tickets = [], []

        def submit():
            t = time.perf_counter()
            tickets.append(gcb.gc_batch_submit(b, *g))
            worst.append(time.perf_counter() - t)

        def refused():
            with pytest.raises(gcb.GcError) as ei:
                gcb.gc_batch_submit(b, g[0], bad)
            assert ei.value.status == -3

        submit()
        run_threads(*[submit] * 6, refused)  # more than the checks that may run at a time
        assert not done.query()  # the GPU was taken all the while
        assert max(worst) < 0.1
        gcb.gc_batch_flush(b)
        assert all(gcb.gc_batch_poll(b, t) == expect for t in tickets)
        t = gcb.gc_batch_submit(b, *g)  # what the checks left behind is taken up again
        gcb.gc_batch_flush(b)
        assert gcb.gc_batch_poll(b, t) == expect
    finally:
        gcb.gc_batch_destroy(b)


@pytest.mark.parametrize("flags", [0, gcb.GC_BATCH_MANUAL])
def test_pinned_memory_is_given_back_without_the_lock(flags):
    # 150 outstanding submissions hold 150 pinned blocks, of which 64 are kept;
    # giving the others back waits for the whole device, here a kernel that sleeps,
    # and must not keep other threads' calls waiting
    import torch
    g = graphgen.er(200, 0.25, 9)  # above 4096 entries: pinned
    expect = batch_count(g)
    b = gcb.gc_batch_create(8 << 30, flags)
    try:
        # not launched one by one as they come: behind one long launch
        first = gcb.gc_batch_submit(b, *graphgen.chung_lu(200000, 3000000, 2.1, 6e6, 30000.0, 3))
        tickets = [gcb.gc_batch_submit(b, *g) for _ in range(150)]
        gcb.gc_batch_flush(b)
        if flags:
            torch.cuda.synchronize()
            torch.cuda._sleep(2_000_000_000)
        else:
            while gcb.gc_batch_poll(b, first, timeout_us=0) is None:
                time.sleep(1e-4)
            torch.cuda._sleep(2_000_000_000)
        done = torch.cuda.Event()
        done.record()
        worst = []

        def others():
            time.sleep(0.05)
            while not done.query() and len(worst) < 50:
                t = time.perf_counter()
                extra = gcb.gc_batch_submit(b, *g)
                assert flags or gcb.gc_batch_poll(b, extra, timeout_us=0) in (None, expect)
                worst.append(time.perf_counter() - t)
                time.sleep(0.005)

        def poll():
            got = gcb.gc_batch_poll_many(b, np.array(tickets, np.uint64))
            assert all(int(v) == e for x in got for v, e in zip(x[:, 0], expect))

        run_threads(poll, others)
        assert len(worst) > 5 and max(worst) < 0.2
    finally:
        gcb.gc_batch_destroy(b)


def test_a_ticket_that_is_never_polled_keeps_no_later_ones():
    import os
    import subprocess
    import sys
    code = """
import ctypes, numpy as np, graphgen, paper_1608_05138_gb300 as gc
class Info(ctypes.Structure):
    _fields_ = [(k, ctypes.c_size_t) for k in 'arena ordblks smblks hblks hblkhd usmblks fsmblks uordblks fordblks keepcost'.split()]
mallinfo2 = ctypes.CDLL(None).mallinfo2
mallinfo2.restype = Info
def held():  # bytes of this thread's heap in use
    return mallinfo2().uordblks + mallinfo2().hblkhd
b = gc.gc_batch_create(8 << 30, gc.GC_BATCH_MANUAL)
first = graphgen.er(30, 0.2, 1)
t0 = gc.gc_batch_submit(b, *first)
G = 100000
nv, vo, eo = np.full(G, 2), np.arange(G + 1) * 3, np.arange(G + 1) * 2
rp, ci = np.tile(np.array([0, 1, 2], np.int32), G), np.tile(np.array([1, 0], np.int32), G)
size = []
for i in range(40):
    t = gc.gc_batch_submit_many(b, nv, vo, eo, rp, ci)
    gc.gc_batch_flush(b)
    x = gc.gc_batch_poll_many(b, t)
    assert (x[:, 0, 0] == 1).all()
    if i in (4, 39):
        size.append(held())
assert size[1] - size[0] < 40 << 20, size
with gc.Graph(*first) as g:
    assert gc.gc_batch_poll(b, t0) == g.count()
try:
    gc.gc_batch_poll(b, t0)
    raise SystemExit('a retired ticket was found')
except gc.GcError:
    pass
gc.gc_batch_destroy(b)
print('ok')
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr


def test_live_handles_keep_no_side_streams():
    # 200 live handles, each counted: a side stream takes 0.57 MB of device memory,
    # and a count of this graph uses two or three
    import torch
    g = graphgen.er(1000, 0.02, 1)
    expect = batch_count(g)
    handles = [gcb.Graph(*g) for _ in range(200)]
    try:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        assert all(h.count() == expect for h in handles)
        assert free - torch.cuda.mem_get_info()[0] < 64 << 20
    finally:
        for h in handles:
            h.close()


def test_a_count_keeps_its_streams_priority():
    # beside a kernel of many short CTAs on a stream of lower priority, a count's
    # kernels get the slots that come free; at equal priority they would wait until
    # all of its CTAs are placed
    import torch
    g = graphgen.chung_lu(60000, 500000, 2.2, 1e6, 3000.0, 3)
    z = torch.full((1 << 29,), 3.3, dtype=torch.float64, device="cuda")
    with gcb.Graph(*g, stream=torch.cuda.Stream(priority=-1)) as h:
        expect = h.count()
        torch.lgamma(z, out=z)  # compiled and warm
        z.fill_(3.3)
        torch.cuda.synchronize()
        t = time.perf_counter()
        torch.lgamma(z, out=z)
        torch.cuda.synchronize()
        alone = time.perf_counter() - t
        z.fill_(3.3)
        torch.cuda.synchronize()
        torch.lgamma(z, out=z)
        done = torch.cuda.Event()
        done.record()
        t = time.perf_counter()
        assert h.count() == expect
        took = time.perf_counter() - t
        assert not done.query()
    assert took < alone / 3


def test_a_count_stays_on_its_streams_part_of_the_gpu():
    # a green context of 16 SMs: a count on its stream takes several times as long
    # as on the whole GPU, and the same counts come out
    import ctypes as C
    import torch
    cu = C.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("no green contexts in this driver")

    class Resource(C.Structure):  # CUdevResource: type, padding, union
        _fields_ = [("type", C.c_int), ("pad", C.c_ubyte * 92), ("sm", C.c_uint), ("rest", C.c_ubyte * 44)]

    torch.zeros(1, device="cuda")
    whole, part, rest = Resource(), Resource(), Resource()
    count, desc, ctx, stream = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    assert cu.cuDeviceGetDevResource(0, C.byref(whole), 1) == 0
    assert cu.cuDevSmResourceSplitByCount(C.byref(part), C.byref(count), C.byref(whole), C.byref(rest), 0, 16) == 0
    assert part.sm == 16
    assert cu.cuDevResourceGenerateDesc(C.byref(desc), C.byref(part), 1) == 0
    assert cu.cuGreenCtxCreate(C.byref(ctx), desc, 0, 1) == 0
    assert cu.cuGreenCtxStreamCreate(C.byref(stream), ctx, 1, 0) == 0
    took = {}
    g = graphgen.chung_lu(100000, 1500000, 2.2, 3e6, 5000.0, 3)
    counts = {}
    try:
        for name, s in (("whole", torch.cuda.Stream().cuda_stream), ("part", stream.value)):
            with gcb.Graph(*g, stream=s) as h:
                times = []
                for _ in range(4):
                    t = time.perf_counter()
                    counts[name] = h.count()
                    times.append(time.perf_counter() - t)
                took[name] = min(times)
    finally:
        torch.cuda.synchronize()
        cu.cuStreamDestroy_v2(stream)
        cu.cuGreenCtxDestroy(ctx)
    assert counts["part"] == counts["whole"]
    assert took["part"] > 3 * took["whole"], took


def test_a_count_with_another_device_current_is_refused():
    import torch
    if torch.cuda.device_count() < 2:
        pytest.skip("needs two devices")
    g = gcb.Graph(*graphgen.er(300, 0.1, 1))
    try:
        x = g.count()
        with torch.cuda.device(1):
            with pytest.raises(gcb.GcError) as ei:
                g.count()
        assert ei.value.status == -8
        assert g.count() == x
    finally:
        g.close()
