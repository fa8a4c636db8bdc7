"""The rules that pick a kernel by the shape of a graph: results on both sides of
each line, and work that follows the shape (a sparse or skewed graph must not
cost what a dense one of its size does)."""
import ctypes as C
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
    (lambda: bipartite(60, 3000), True),            # rows of hubs, read once for every leaf
    (lambda: hubs(200, 2000, 5), True),
    (lambda: hubs(60, 3000, 4), True),
    (lambda: bipartite(550, 700), True),             # dense, but without a triangle
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


def triangles(rp, ci):
    import torch
    a, b = torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda()
    out = torch.full((len(ci),), -1, dtype=torch.int32, device="cuda")
    gcb.gc_edge_triangles_noalloc(a, b, out)
    return out.cpu().numpy()


@pytest.mark.parametrize("make", [
    lambda: graphgen.er(1024, 0.05, 1),      # the largest graph of one kernel
    lambda: graphgen.er(1025, 0.05, 1),      # picked on the device: one kernel
    lambda: graphgen.er(4096, 0.02, 1),
    lambda: graphgen.er(4097, 0.02, 1),      # beyond
    lambda: graphs.complete(64),             # rows of 63 entries: end to end
    lambda: graphs.complete(66),             # and of 65: one at a time
    lambda: graphs.star(1000),
    lambda: graphs.star(4095),               # picked: the kernels of larger graphs
    lambda: bipartite(60, 2000),
    lambda: hubs(20, 3000, 4),
    lambda: graphs.csr(3000, [(7, 2999)]),
])
def test_noalloc_kernel_by_size_and_shape(make):
    rp, ci = make()
    t = oracle.count(rp, ci)["per_edge"][:, 0]
    uv = oracle.edges(rp, ci)
    n = len(rp) - 1
    rows = np.repeat(np.arange(n, dtype=np.int64), np.diff(rp))
    at = np.searchsorted(uv[:, 0].astype(np.int64) * n + uv[:, 1],
                         np.minimum(rows, ci) * n + np.maximum(rows, ci))
    np.testing.assert_array_equal(triangles(rp, ci), t[at].astype(np.int32))


@pytest.mark.parametrize("n", [300, 1500, 3000])
@pytest.mark.parametrize("skew", [False, True])
def test_noalloc_rows_that_break_the_rules_by_size(n, skew):
    # as test_noalloc_rows_that_break_the_rules, for every kernel that a size and shape pick
    rng = np.random.default_rng(n + skew)
    rp, ci = graphgen.chung_lu(n, 9 * n, 2.1, 18.0 * n, n - 1.0, 5) if skew else graphgen.er(n, 20.0 / n, 5)
    ci = ci.copy()
    for x in rng.choice(n, 60, replace=False):
        row = ci[rp[x]:rp[x + 1]]
        if len(row) >= 3:
            k = rng.integers(0, 4)
            if k == 0:
                rng.shuffle(row)
            elif k == 1:
                row[0] = row[-1]
            elif k == 2:
                row[rng.integers(0, len(row))] = rng.choice([-1, n, 2**31 - 1, -2**31])
            else:
                row[rng.integers(0, len(row))] = x
    rows = [ci[rp[x]:rp[x + 1]].tolist() for x in range(n)]
    sets = [set(r) for r in rows]
    expect = [sum(0 <= w < n and w in sets[x] for w in rows[y]) if 0 <= y < n else 0 for x in range(n) for y in rows[x]]
    np.testing.assert_array_equal(triangles(rp, ci), np.array(expect, np.int32))


def test_noalloc_small_call_is_one_kernel_and_can_be_captured():
    # the smallest calls are launches; and every launch sequence replays as a graph
    import torch
    cu = C.CDLL("libcuda.so.1")
    for (rp, ci), most in ((graphgen.er(500, 0.1, 3), 1), (graphgen.er(3000, 0.01, 3), 6), (graphgen.er(9000, 0.003, 3), 6)):
        expect = triangles(rp, ci)  # also the first call, which looks the array up
        a, b = torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda()
        out = torch.full((len(ci),), -1, dtype=torch.int32, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        graph, ex, count = C.c_void_p(), C.c_void_p(), C.c_size_t()
        torch.cuda.synchronize()
        h = C.c_void_p(s.cuda_stream)
        n = C.c_int32(len(rp) - 1)
        assert cu.cuStreamBeginCapture_v2(h, 1) == 0
        st = gcb.lib().gc_edge_triangles_noalloc(n, C.c_void_p(a.data_ptr()), C.c_void_p(b.data_ptr()),
                                                 C.c_void_p(out.data_ptr()), h)
        assert cu.cuStreamEndCapture(h, C.byref(graph)) == 0 and st == 0
        assert cu.cuGraphGetNodes(graph, None, C.byref(count)) == 0
        assert cu.cuGraphInstantiateWithFlags(C.byref(ex), graph, C.c_ulonglong(0)) == 0
        for _ in range(2):
            out.fill_(-1)
            torch.cuda.synchronize()
            assert cu.cuGraphLaunch(ex, h) == 0
            torch.cuda.synchronize()
            np.testing.assert_array_equal(out.cpu().numpy(), expect)
        cu.cuGraphExecDestroy(ex)
        cu.cuGraphDestroy(graph)
        assert 1 <= count.value <= most


def test_noalloc_slots_beyond_2_to_the_30():
    # 950 complete graphs on 1100 vertices: 1.15e9 slots, so that the sum of two of
    # them, as a binary search forms it, passes 2^31
    import torch
    k, copies = 1100, 950
    v = torch.arange(k, dtype=torch.int32, device="cuda")
    block = v.repeat(k, 1)[~torch.eye(k, dtype=torch.bool, device="cuda")]
    ci = (block[None, :] + (torch.arange(copies, dtype=torch.int32, device="cuda") * k)[:, None]).reshape(-1)
    rp = (torch.arange(copies * k + 1, dtype=torch.int64, device="cuda") * (k - 1)).to(torch.int32)
    assert ci.numel() > 1 << 30
    out = torch.full_like(ci, -1)
    gcb.gc_edge_triangles_noalloc(rp, ci, out)
    assert bool((out == k - 2).all())
    del ci, out
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n, sizes", [
    # rows of one more and one less than a warp's and a CTA's, of runs that a lane, a
    # warp and a CTA reads; the last n of four CTAs an SM and the first of larger ones
    (358400, [17, 64, 65, 66, 128, 129, 130, 131, 256, 257, 258, 600, 2048, 2049, 2050, 2600]),
    (358432, [17, 64, 65, 66, 128, 129, 130, 131, 256, 257, 258, 600, 2048, 2049, 2050, 2600]),
    (1 << 20, [17, 64, 65, 66, 128, 129, 130, 131, 256, 257, 258, 600, 2048, 2049, 2050, 2600]),
    (131073, [2100] * 62),  # 2^28 entries: more of a part's runs than its CTA can list
])
def test_noalloc_long_rows_by_number_of_vertices(n, sizes):
    # disjoint complete graphs after isolated vertices
    import torch
    ks = torch.tensor(sizes, device="cuda")
    k = torch.cat([torch.zeros(n - sum(sizes), dtype=torch.long, device="cuda"), torch.repeat_interleave(ks, ks)])
    rp = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rp[1:] = torch.cumsum((k - 1).clamp(min=0), 0)
    ci, at = [], n - sum(sizes)
    for s in sizes:
        v = torch.arange(s, dtype=torch.int32, device="cuda")
        ci.append(v.repeat(s, 1)[~torch.eye(s, dtype=torch.bool, device="cuda")] + at)
        at += s
    out = torch.full((int(rp[-1]),), -1, dtype=torch.int32, device="cuda")
    gcb.gc_edge_triangles_noalloc(rp, torch.cat(ci), out)
    assert torch.equal(out, torch.repeat_interleave(k - 2, (k - 1).clamp(min=0)).to(torch.int32))
    del ci, out, k
    torch.cuda.empty_cache()


def test_noalloc_last_row_of_as_many_parts_as_there_are():
    # not symmetric: the last of 2^20 vertices has 1 048 420 entries, its last part
    # the largest number a list entry can hold; all other rows are empty
    import torch
    n, d = 1 << 20, 4095 * 256 + 100
    rp = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    rp[n] = d
    out = torch.full((d,), -7, dtype=torch.int32, device="cuda")
    gcb.gc_edge_triangles_noalloc(rp, torch.arange(d, dtype=torch.int32, device="cuda"), out)
    assert bool((out == 0).all())


def test_hub_rows_beyond_2_to_the_30_slots():
    # a circulant graph of 67.2M vertices of degree 16, and beside it a hub joined to
    # 2000 vertices that share 60 000 others: the highest degrees, so that their
    # slots are the last ones. The connected graphlets of both add up.
    n0, half = 67_200_000, 8
    off = np.r_[-half:0, 1:half + 1].astype(np.int32)
    rng = np.random.default_rng(1)
    shared = np.stack([1 + rng.integers(0, 2000, 60000 * 32), np.repeat(2001 + np.arange(60000), 32)], 1)
    small_rp, small_ci = graphs.csr_large(62001, np.concatenate([np.stack([np.zeros(2000, int), 1 + np.arange(2000)], 1),
                                                                 shared]))
    assert 16 * n0 > 1 << 30
    ci = np.empty(16 * n0 + len(small_ci), np.int32)
    body = ci[:16 * n0].reshape(n0, 16)
    np.add(np.arange(n0, dtype=np.int32)[:, None], off, out=body)
    for x in list(range(half)) + list(range(n0 - half, n0)):
        body[x] = np.sort((x + off.astype(np.int64)) % n0)
    ci[16 * n0:] = small_ci + n0
    rp = np.concatenate([np.arange(n0, dtype=np.int64) * 16, 16 * n0 + small_rp.astype(np.int64)]).astype(np.int32)
    with gcb.Graph(rp, ci) as g:
        X = g.count()
        w = g.work_counts()
    del ci, body
    gcb.gc_release_cached_memory()
    a = oracle.count(*graphs.csr(1000, [(x, (x + d) % 1000) for x in range(1000) for d in range(1, half + 1)]))["X"]
    with gcb.Graph(small_rp, small_ci) as g:
        b = g.count()
    for i in (2, 3, 6, 7, 8, 9, 10, 11):  # X_3, X_4 and X_7 .. X_12
        assert X[i] == a[i] * (n0 // 1000) + b[i], i + 1
    assert w["c_hub_jobs"] > 0


# ---- the paths that small graphs no longer take by themselves ----

def padded(g, n):
    """The graph with isolated vertices added up to n: beyond 4096, passes T, C and K count it."""
    rp, ci = g
    return np.concatenate([rp, np.full(n + 1 - len(rp), rp[-1], np.int32)]), ci


def by_passes(g, scans, times=2):
    """Counts the graph, padded beyond 4096 vertices, against the oracle; scans: whether pass K scans in the last
    count, or replays the lists that pass T kept."""
    rp, ci = padded(g, max(len(g[0]) - 1, 4200))
    o = oracle.count(rp, ci)
    with gcb.Graph(rp, ci) as h:
        for _ in range(times):
            pe = np.zeros((h.m, 13), np.uint64)
            assert h.count(pe) == o["X"]
            np.testing.assert_array_equal(pe, o["per_edge"])
        w = h.work_counts()
    assert w["t_members"] > 0 and w["t_triangles"] == w["k_local_edges"] == o["X"][2]
    assert (w["k_scan"] > 0) == scans


@pytest.mark.parametrize("make", [
    lambda: graphgen.chung_lu(3000, 15000, 2.1, 30000.0, 800.0, 5),
    lambda: graphgen.rmat(12, 16, 0.57, 0.19, 0.19, 6),
    graphgen.config_er_dense,
    lambda: graphs.complete(300),
])
def test_replayed_triangle_lists_of_every_tier(make):
    by_passes(make(), scans=False, times=3)


def test_replayed_triangle_lists_of_the_global_tier():
    # out-degrees a little above 1024, lists of fewer than 2^19 edges; x3, x7 and x10
    # do not change with isolated vertices, and without them the graph takes the rows
    g = graphgen.er(1170, 0.915, 41)
    cols = []
    for h in (padded(g, 4200), g):
        with gcb.Graph(*h) as G:
            for _ in range(2):
                pe = np.zeros((G.m, 13), np.uint64)
                G.count(pe)
                cols.append(pe[:, [0, 3, 4]])
            w = G.work_counts()
        assert (w["t_members"] > 0) == (len(h[0]) > 4096)
        if w["t_members"]:
            assert w["k_scan"] == 0
    for c in cols[1:]:
        np.testing.assert_array_equal(c, cols[0])
    uv = oracle.edges(*g)
    pick = np.random.default_rng(1).choice(len(uv), 100, replace=False)
    np.testing.assert_array_equal(cols[0][pick], oracle.count_sample(*g, pick)[:, [0, 3, 4]])


def run_with_env(call, **env):
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", f"import tests.test_gpu_routes as t; t.{call}; print('ok')"], cwd=root,
                       env=dict(os.environ, PYTHONPATH=root, **env), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "ok" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("env", [{"GC_K_LIST_CAP": "64"}, {"GC_T_LIST_CAP": "5000"}])
def test_pass_k_scans_again_where_lists_are_short(env):
    run_with_env("by_passes(t.graphgen.rmat(12, 16, 0.57, 0.19, 0.19, 29), scans=True)", **env)
    run_with_env("by_passes(t.graphgen.config_er_dense(), scans=True)", **env)


@pytest.mark.parametrize("n", [1025, 1026])  # out-degrees up to 1024: bit rows; 1025: not
def test_complete_graphs_at_the_limit_of_the_bit_rows(n):
    m = n * (n - 1) // 2
    with gcb.Graph(*graphgen.er(n, 1.0, 1)) as g:
        pe = np.zeros((g.m, 13), np.uint64)
        assert g.count(pe) == [m, 0, comb(n, 3), 0, 0, 0, comb(n, 4)] + [0] * 10
    row = [n - 2, 0, 0, comb(n - 2, 2), 0, comb(n - 2, 2), 0, 0, 0, 0, m - 2 * (n - 1) + 1, 0, 0]
    assert (pe == np.array(row, np.uint64)).all()


@pytest.mark.parametrize("n", [2047, 2048])
def test_bit_rows_of_the_largest_graphs(n):
    # all 64 words; 60 vertices joined to all, any two of which share more than 1024
    # neighbours (the highest plane of the counts), among others of about 950
    from tests.test_gpu_parity import _sampled_check
    rp, ci = graphgen.er(n, 0.44, 3)
    rows = np.repeat(np.arange(n), np.diff(rp))
    up = rows < ci
    u, v = np.meshgrid(np.arange(60), np.arange(n), indexing="ij")
    e = np.concatenate([np.stack([rows[up], ci[up]], 1), np.stack([u.ravel(), v.ravel()], 1)[(u != v).ravel()]])
    rp, ci = graphs.csr_large(n, e)
    with gcb.Graph(rp, ci) as g:
        g.count()
        w = g.work_counts()
    assert w["t_members"] == 0 and w["launches"] == 4  # rows, cliques, finish, derive
    _sampled_check(rp, ci, k=100, seed=n)


# ---- the hub kernel's counters at the limits of their fields ----

def hub_segments(degrees, tab):
    """Counters per word of the segments that the ids of these degrees (ascending) are cut into: each takes the width
    that reaches furthest, up to the end of its block or of the ids whose counts fit it."""
    bound = [int(np.searchsorted(degrees, d)) for d in (2, 4, 16, 256, 65536)]
    end, lo, word, out = len(degrees), bound[0], 0, []
    while lo < end:
        hi, lg = lo, 0
        for k in range(5):
            to = min(end if k == 0 else bound[5 - k], lo + ((tab - word) << k))
            if to > hi:
                hi, lg = to, k
        out.append((lo, hi, 1 << lg))
        word += (hi - lo + (1 << lg) - 1) >> lg
        if tab - word < tab // 16 or hi == end:
            word = 0
        lo = hi
    return out


def check_field_limits():
    # a hub joined to 3000 vertices x; others, o, whose neighbours are all x, so that
    # the hub's count of o is its degree: 2, 3 / 4, 15 / 16, 255 / 256, so many of each
    # that the ids of a class reach further than a block of wider counters. No triangle:
    # every 4-cycle is induced, and x10 of (x, y) is the sum over the other neighbours
    # x' of y of the common neighbours of x and x' without y.
    import torch
    nx, rng = 3000, np.random.default_rng(7)
    deg = np.repeat([2, 3, 4, 15, 16, 255, 256], [20000, 20000, 8000, 2000, 10000, 300, 4300])
    key = rng.random((2000, nx))
    rows, at = [], 0
    for d in deg:  # d of the nx, by a random row of keys, shifted
        rows.append(np.argpartition(np.roll(key[at % 2000], at), d - 1)[:d] if d > 4 else rng.choice(nx, d, replace=False))
        at += 1
    x = np.concatenate([np.arange(nx)] + rows)
    y = nx + np.concatenate([np.zeros(nx, int), np.repeat(1 + np.arange(len(deg)), deg)])
    rp, ci = graphs.csr_large(nx + 1 + len(deg), np.stack([x, y], 1))
    degrees = np.sort(np.diff(rp))
    assert degrees[-1] == nx  # the hub is the last
    segments = hub_segments(degrees, 4096)
    for d, counters in ((3, 16), (15, 8), (255, 4), (256, 2)):  # the largest counts of a field, and one more bit
        i = int(np.searchsorted(degrees, d, side="right")) - 1 if d != 256 else int(np.searchsorted(degrees, d))
        assert [c for lo, hi, c in segments if lo <= i < hi] == [counters], (d, segments)
    with gcb.Graph(rp, ci) as g:
        pe = np.zeros((g.m, 13), np.uint64)
        X = g.count(pe)
        uv = g.edges().astype(np.int64)
        w = g.work_counts()
    assert w["c_heavy_wedges"] >= deg.sum()
    a = torch.zeros((nx, 1 + len(deg)), dtype=torch.float64, device="cuda")
    a[torch.from_numpy(x).cuda(), torch.from_numpy(y - nx).cuda()] = 1.0
    q = a @ a.T - 1.0
    q.fill_diagonal_(0.0)
    pairs = (q + 1.0).cpu().numpy()
    x10 = (q @ a).cpu().numpy()[uv[:, 0], uv[:, 1] - nx]
    np.testing.assert_array_equal(pe[:, 4].astype(np.int64), x10.astype(np.int64))
    assert not pe[:, 0].any()
    i = np.triu_indices(nx, 1)
    assert X[9] == int((pairs[i] * (pairs[i] - 1) / 2).sum())


def test_hub_counters_at_the_limits_of_every_field():
    run_with_env("check_field_limits()", GC_HUB_TAB_WORDS="4096")


# ---- induced counts: rows of more than 4096 entries ----

@pytest.mark.parametrize("make", [
    lambda: graphs.star(4096),               # a warp's longest row
    lambda: graphs.star(4097),               # a CTA's shortest
    lambda: hubs(2, 5000, 1),
])
def test_induced_counts_beside_long_rows(make):
    from tests.test_gpu_induced import assert_induced_parity
    assert_induced_parity(*make())


def test_induced_counts_do_not_wait_for_one_warp():
    # the sums over the neighbours of a star's centre were one warp's, 0.64 ms
    import torch
    with gcb.Graph(*graphs.csr_large(100001, [(0, x) for x in range(1, 100001)])) as g:
        n = g.n
        ind = torch.zeros((g.m, 10), dtype=torch.int64, device="cuda")
        took = []
        for _ in range(5):
            g.count_induced(ind)
            took.append(g.phase_ms()["induced_columns"])
    ind = ind.cpu().numpy()
    assert (ind[:, 4] == comb(n - 2, 2)).all() and not ind[:, [0, 1, 2, 3, 5, 6, 7, 8, 9]].any()
    assert min(took) < 0.3
