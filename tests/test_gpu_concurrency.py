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
