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
