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
    rp, ci = graphgen.er(200000, 4e-4, 5)  # 8M entries: 64 MB of CSR
    bad = ci.copy()
    x = int(np.flatnonzero(np.diff(rp) >= 3)[0])
    bad[rp[x]] = bad[rp[x] + 1]
    need = 44 * 200000 + 32 * (len(ci) // 2) + 1024 + 2 * 152 * 200000 * 4
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
        assert free - torch.cuda.mem_get_info()[0] < 16 << 20
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
