"""The allocation-free triangle entry point against the regular one.

gc_edge_triangles_noalloc serves callers that cannot allocate device memory:
it reads a device CSR in place and keeps its only scratch in a fixed
file-scope device array. Here it is called through the C ABI twice in a row
(the array keeps the previous call's contents, so the second call checks that
each call starts clean) and its per-slot counts must equal column 0 (|T|) of
gc_count_edge_graphlets for the same edges, and |T| of the CPU oracle,
exactly (integer counts). A call after the first one must leave the device's
free memory and torch's allocated bytes unchanged. This file is collected
last on purpose.
"""
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


def _slot_edge_ids(rp, ci, uv):
    """Edge id (row of the edge list uv, u < v) behind every CSR slot."""
    n = len(rp) - 1
    key = uv[:, 0].astype(np.int64) * n + uv[:, 1]
    rows = np.repeat(np.arange(n, dtype=np.int64), np.diff(rp))
    cols = ci.astype(np.int64)
    return np.searchsorted(key, np.minimum(rows, cols) * n + np.maximum(rows, cols))


def _oracle_per_slot(rp, ci):
    """|T| of the edge behind every CSR slot, from the CPU oracle."""
    t = oracle.count(rp, ci)["per_edge"][:, 0]
    return t[_slot_edge_ids(rp, ci, oracle.edges(rp, ci))].astype(np.int32)


def _expected_per_slot(rp, ci):
    """|T| of the edge behind every CSR slot, from the regular entry point."""
    with gcb.Graph(rp, ci) as g:
        pe = np.zeros((g.m, 13), np.uint64)
        g.count(pe)
        uv = g.edges()
    return pe[_slot_edge_ids(rp, ci, uv), 0].astype(np.int32)


@pytest.mark.parametrize("make", [
    lambda: graphgen.chung_lu(50000, 400000, 2.1, 800000.0, 4000.0, 61),
    lambda: graphgen.er(3000, 0.05, 62),
    lambda: graphs.complete(40),
    lambda: graphs.star(500),
])
def test_noalloc_matches_regular_entry_point_twice(make):
    import torch
    rp, ci = make()
    expect = _expected_per_slot(rp, ci)
    np.testing.assert_array_equal(expect, _oracle_per_slot(rp, ci))
    d_rp = torch.from_numpy(rp).cuda()
    d_ci = torch.from_numpy(ci).cuda()
    stream = torch.cuda.current_stream()
    for _ in range(2):
        out = torch.full((len(ci),), -1, dtype=torch.int32, device="cuda")
        gcb.gc_edge_triangles_noalloc(d_rp, d_ci, out, stream=stream)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), expect)


@pytest.mark.parametrize("make", [
    lambda: graphs.complete(128),          # rows of 127 entries: the longest a warp takes
    lambda: graphs.complete(131),          # rows of 130: a CTA's
    lambda: graphgen.chung_lu(1 << 20, 300000, 2.1, 600000.0, 3000.0, 64),  # the largest bitmap
    lambda: graphs.csr(70, [(3, 40)]),     # one edge, a partial bitmap word
])
def test_noalloc_row_lengths(make):
    import torch
    rp, ci = make()
    d_rp, d_ci = torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda()
    out = torch.full((len(ci),), -1, dtype=torch.int32, device="cuda")
    gcb.gc_edge_triangles_noalloc(d_rp, d_ci, out)
    np.testing.assert_array_equal(out.cpu().numpy(), _oracle_per_slot(rp, ci))


@pytest.mark.parametrize("k, copies, pad", [
    (33, 3, 0), (34, 3, 0),                    # rows of 32, 33 entries, fewer than 2^18 in all
    (129, 1, 0), (130, 1, 0),                  # one part of 128 slots, and one slot more
    (65, 70, 0), (66, 70, 0),                  # 64, 65 of fewer than 2^20
    (257, 5, 0), (258, 5, 0),                  # a part of 256, and one slot more
    (129, 70, 0), (130, 70, 0),                # 128, 129 of 2^20 or more
    (513, 5, 0), (514, 5, 0),                  # a part of 512, and one slot more
    (66, 70, 1 << 17), (130, 70, 1 << 17),     # long and short rows in kernels of their own
])
def test_noalloc_split_of_the_rows(k, copies, pad):
    # disjoint complete graphs on k vertices: k - 2 triangles on every edge; and
    # as many isolated vertices as asked for
    import torch
    v = np.arange(k, dtype=np.int32)
    block = np.array([np.delete(v, x) for x in range(k)], np.int32).ravel()
    ci = np.concatenate([block + c * k for c in range(copies)]).astype(np.int32)
    rp = np.concatenate([np.arange(copies * k + 1) * (k - 1), np.full(pad, len(ci))]).astype(np.int32)
    out = torch.full((len(ci),), -1, dtype=torch.int32, device="cuda")
    gcb.gc_edge_triangles_noalloc(torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), out)
    assert (out == k - 2).all()


@pytest.mark.parametrize("seed", range(4))
def test_noalloc_rows_that_break_the_rules(seed):
    # not validated, but safe and by the definition: tri[p] of (x, y) is the
    # number of entries of row y in [0, n) that are in row x; 0 for y outside
    import torch
    rng = np.random.default_rng(seed)
    n = 300
    rp, ci = graphgen.chung_lu(n, 4000, 2.3, 8000.0, 200.0, 70 + seed)
    ci = ci.copy()
    for x in rng.choice(n, 40, replace=False):
        row = ci[rp[x]:rp[x + 1]]
        if len(row) < 3:
            continue
        kind = rng.integers(0, 5)
        if kind == 0:
            rng.shuffle(row)                              # unsorted
        elif kind == 1:
            row[0] = row[-1]                              # a neighbour twice, one reverse missing
        elif kind == 2:
            row[rng.integers(0, len(row))] = rng.choice([-1, n, 2**31 - 1, -2**31])
        elif kind == 3:
            row[rng.integers(0, len(row))] = x            # self-loop
        else:
            free = np.setdiff1d(np.arange(n), np.append(row, x))
            if len(free):
                row[0] = free[0]                          # sorted or not, asymmetric
                row.sort()
    rows = [ci[rp[x]:rp[x + 1]] for x in range(n)]
    sets = [set(r.tolist()) for r in rows]
    expect = [sum(0 <= w < n and w in sets[x] for w in rows[y].tolist()) if 0 <= y < n else 0
              for x in range(n) for y in rows[x].tolist()]
    out = torch.full((len(ci),), -7, dtype=torch.int32, device="cuda")
    gcb.gc_edge_triangles_noalloc(torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), out)
    np.testing.assert_array_equal(out.cpu().numpy(), np.array(expect, np.int32))


def test_noalloc_rejects_graphs_above_its_limit():
    import torch
    n = (1 << 20) + 1
    d_rp = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    d_ci = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.zeros(1, dtype=torch.int32, device="cuda")
    with pytest.raises(gcb.GcError) as ei:
        gcb.gc_edge_triangles_noalloc(d_rp, d_ci, out)
    assert ei.value.status == -9
    assert "limit" in str(ei.value)


def test_noalloc_call_allocates_nothing():
    import torch
    rp, ci = graphgen.er(3000, 0.05, 63)
    d_rp = torch.from_numpy(rp).cuda()
    d_ci = torch.from_numpy(ci).cuda()
    out = torch.zeros(len(ci), dtype=torch.int32, device="cuda")
    gcb.gc_edge_triangles_noalloc(d_rp, d_ci, out)  # first call: module and symbol set-up
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    alloc0 = torch.cuda.memory_allocated()
    gcb.gc_edge_triangles_noalloc(d_rp, d_ci, out)
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert torch.cuda.memory_allocated() == alloc0
    assert free1 == free0
    np.testing.assert_array_equal(out.cpu().numpy(), _oracle_per_slot(rp, ci))
