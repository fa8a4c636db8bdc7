"""The rules that pick a kernel by the shape of a graph: results on both sides of
each line, and work that follows the shape (a sparse or skewed graph must not
cost what a dense one of its size does)."""
from math import comb

import numpy as np
import pytest

import graphgen
import oracle
import paper_1608_05138_gb300 as gcb
from tests import graphs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1608_05138_gb300 import build
    build.build()


def bipartite(a, b):
    u, v = np.meshgrid(np.arange(a), a + np.arange(b), indexing="ij")
    return graphs.csr_large(a + b, zip(u.ravel(), v.ravel()))


def hubs(h, n, d, seed=1):
    """h vertices joined to all the others, which have d random edges each."""
    rng = np.random.default_rng(seed)
    u, v = np.meshgrid(np.arange(h), np.arange(h, n), indexing="ij")
    e = np.concatenate([np.stack([u.ravel(), v.ravel()], 1), rng.integers(h, n, ((n - h) * d, 2))])
    return graphs.csr_large(n, e[e[:, 0] != e[:, 1]])


def wide(n, k, edges, seed):
    """Vertex 0 joined to 1 .. k, and so many random edges among those: an H_0 of few edges."""
    rng = np.random.default_rng(seed)
    e = np.concatenate([np.stack([np.zeros(k, int), 1 + np.arange(k)], 1), 1 + rng.integers(0, k, (edges, 2))])
    clique = [(a, b) for a in range(1, 7) for b in range(a + 1, 7)]  # some 4-cliques with certainty
    return graphs.csr_large(n, list(e[e[:, 0] != e[:, 1]]) + clique)


def batch_counts(gs, n_max=1024):
    b = gcb.gc_batch_create(8 << 30, gcb.GC_BATCH_MANUAL)
    try:
        gcb.gc_batch_set_param(b, gcb.GC_PARAM_SMALL_N_MAX, n_max)
        t = [gcb.gc_batch_submit(b, *g) for g in gs]
        gcb.gc_batch_flush(b)
        X = [gcb.gc_batch_poll(b, k) for k in t]
        return X, gcb.gc_batch_last_stats(b)["small_sequence_ms"]
    finally:
        gcb.gc_batch_destroy(b)


@pytest.mark.parametrize("copies", [1, 600])  # one graph is cut into parts, many are not
def test_small_graphs_of_every_size_and_shape(copies):
    # four vertices of a warp at a time from 4 * 16 vertices a part; neighbourhoods
    # without edges, of few (counted edge by edge) and of many (packed)
    gs = [graphs.empty(1), graphs.empty(5), graphs.star(1023), graphs.star(64), bipartite(10, 990), bipartite(3, 60),
          wide(1024, 1022, 300, 1), wide(1000, 999, 3000, 2), wide(200, 180, 30, 3), wide(70, 60, 400, 4),
          hubs(10, 500, 2), graphs.complete(67), graphs.cycle(1024)]
    gs += [graphgen.er(n, 0.1, n) for n in (61, 62, 63, 64, 65, 66, 67, 127, 129, 255, 257, 509, 513, 1021, 1023)]
    X, _ = batch_counts(gs + [graphs.cycle(9)] * (copies - 1))
    for g, x in zip(gs, X):
        assert x == oracle.count(*g, per_edge=False)["X"]


def test_small_complete_graph_has_the_largest_sums():
    n = 1024
    X, _ = batch_counts([graphgen.er(n, 1.0, 1)])
    m = n * (n - 1) // 2
    assert X[0] == [m, 0, comb(n, 3), 0, 0, 0, comb(n, 4)] + [0] * 10


def test_small_graphs_without_4_cliques_cost_what_sparse_ones_do():
    # K(10, 990) has ten neighbourhoods of 990 members without an edge; packing
    # them took four times what a sparse graph of the size takes
    t = {}
    for name, g in (("sparse", graphgen.er(1000, 0.02, 1)), ("bipartite", bipartite(10, 990))):
        t[name] = min(batch_counts([g] * 1000)[1] for _ in range(3))
    assert t["bipartite"] < 2 * t["sparse"]


# (graph, whether passes T and C count it)
@pytest.mark.parametrize("make,passes", [
    (lambda: graphgen.er(2000, 0.01, 1), False),     # rows of common neighbours
    (lambda: graphgen.er(3000, 0.02, 1), False),
    (lambda: hubs(5, 3000, 3), False),
    (lambda: graphgen.er(700, 0.2, 1), False),       # bit rows
    (lambda: bipartite(60, 240), False),             # out-degrees of at most 256, without a triangle
    (lambda: bipartite(150, 3900), True),            # rows of hubs, read once for every leaf
    (lambda: hubs(200, 2000, 5), True),
    (lambda: hubs(120, 4000, 4), True),
    (lambda: bipartite(900, 1100), True),            # dense, but without a triangle
])
def test_route_of_graphs_up_to_4096_vertices(make, passes):
    rp, ci = make()
    with gcb.Graph(rp, ci) as g:
        pe = np.zeros((g.m, 13), np.uint64)
        X = g.count(pe)
        w = g.work_counts()
        pe2 = np.zeros((g.m, 13), np.uint64)
        assert g.count(pe2) == X
    o = oracle.count(rp, ci)
    np.testing.assert_array_equal(pe, o["per_edge"])
    np.testing.assert_array_equal(pe2, o["per_edge"])
    assert X == o["X"]
    assert (w["t_members"] > 0) == passes
