"""The workloads this library's speed is judged on.

Every case is work that a program gives the library through its public entry
points (paper_1608_05138_gb300, the same names as the C ABI of include/gc.h):
counts of an uploaded graph, the whole call from a host CSR to rows on the
host, batches of small graphs, a mixed request load, and the triangle step on
a device CSR. Graphs are drawn on the GPU from the seed alone, with the three
generators of the repository's configurations (Erdos-Renyi, Chung-Lu, R-MAT).
An Erdos-Renyi or Chung-Lu or R-MAT graph of a case always has exactly m
edges, so that outputs have the same shape for every seed.

    listed()             the listed cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs and handles a program holds before the call
    run(state)           one pass
    work(case)           the bytes a pass cannot do without
    exact(case, seed)    what run() returns, by dense matrices, for small graphs
"""
import math

import numpy as np
import torch

import paper_1608_05138_gb300 as gc

DEV = "cuda"


def listed():
    return [
        # The smallest whole-graph call of use: one sparse random graph of a few thousand vertices (the
        # repository's ER-2000 configuration). Launches and host work count.
        {"name": "er_2000", "kind": "count", "gen": "er", "n": 2000, "m": 20000},
        # A small dense graph: the 1K-vertex / 150K-edge shape of the paper's GPU comparison. Cliques dominate.
        {"name": "dense_1k", "kind": "count", "gen": "er", "n": 1000, "m": 150000},
        # An ordinary power-law network of half a million edges, sizes odd, as a user's own data has.
        {"name": "chung_lu_63k", "kind": "count", "gen": "chung_lu", "n": 62501, "m": 500009, "gamma": 2.3},
        # The Chung-Lu configuration: 1M vertices, 10M edges, exponent 2.1, degrees capped at 50 000.
        {"name": "chung_lu_1m", "kind": "count", "gen": "chung_lu", "n": 1000000, "m": 10000000, "gamma": 2.1},
        # The R-MAT configuration the headline is quoted on: scale 22, edge factor 16, 64M distinct edges.
        {"name": "rmat_22", "kind": "count", "gen": "rmat", "n": 1 << 22, "m": 64000000},
        # The per-edge induced counts besides the 13 columns, on a graph of 4M edges.
        {"name": "induced_rmat_18", "kind": "induced", "gen": "rmat", "n": 1 << 18, "m": 3800000},
        # From the caller's host CSR to rows in pinned host memory: upload, count, free, as a program that
        # counts each graph once does it.
        {"name": "whole_rmat_20", "kind": "whole", "gen": "rmat", "n": 1 << 20, "m": 15600000},
        # The same for a small sparse graph, where the upload's fixed work is most of the call.
        {"name": "whole_chung_lu_20k", "kind": "whole", "gen": "chung_lu", "n": 20011, "m": 100003, "gamma": 2.5},
        # The batched form: many graphs of 20 to 500 vertices, half Erdos-Renyi, half Chung-Lu, in one submission.
        {"name": "batch_20000", "kind": "batch", "graphs": 20000, "n_lo": 20, "n_hi": 500},
        # A small batch, where the latency of the submission and of one launch counts.
        {"name": "batch_48", "kind": "batch", "graphs": 48, "n_lo": 20, "n_hi": 500},
        # The serving form: requests of Chung-Lu graphs, edges log-uniform from 1 000 to 2M, submitted one by
        # one to a continuously batching runtime with a 120 GB budget.
        {"name": "serve_40", "kind": "serve", "graphs": 40, "m_lo": 1000, "m_hi": 2000000},
        # The allocation-free triangle step on a device CSR of a social-network-like graph.
        {"name": "triangles_100k", "kind": "triangles", "gen": "chung_lu", "n": 100003, "m": 1000003, "gamma": 2.3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, m_lo, m_hi):
    """A generator with sizes of its own range: m log-uniform, the mean degree as in the listed cases."""
    gen = rng.choice(["er", "chung_lu", "chung_lu", "rmat"])
    m = _log_int(rng, m_lo, m_hi)
    if gen == "rmat":  # edge factor 12 to 18, as R-MAT graphs are made
        scale = min(22, max(10, int(round(math.log2(m / 15.3)))))
        return {"gen": "rmat", "n": 1 << scale, "m": min(m, 15 << scale)}
    if gen == "er":  # from sparse (mean degree 8) to dense (density 0.4)
        m = min(m, 2000000)
        n_dense = math.sqrt(2 * m / 0.4)
        return {"gen": "er", "n": _log_int(rng, n_dense, max(n_dense + 1, m / 4)), "m": m}
    m = min(m, 10000000)
    return {"gen": "chung_lu", "n": _log_int(rng, m / 10, m / 5), "m": m, "gamma": round(rng.uniform(2.1, 2.5), 2)}


def draw(rng):
    kind = rng.choice(["count", "count", "count", "induced", "whole", "whole", "batch", "batch", "serve", "triangles"])
    if kind == "batch":
        return {"kind": "batch", "graphs": _log_int(rng, 32, 20000), "n_lo": 20, "n_hi": rng.randint(100, 500)}
    if kind == "serve":
        return {"kind": "serve", "graphs": rng.randint(4, 40), "m_lo": 1000, "m_hi": 2000000}
    if kind == "triangles":
        m = _log_int(rng, 20000, 1000000)
        return {"kind": "triangles", "gen": "chung_lu", "n": _log_int(rng, m / 10, m / 5), "m": m,
                "gamma": round(rng.uniform(2.3, 2.7), 2)}
    top = {"count": 60000000, "induced": 4000000, "whole": 15000000}[kind]
    return {"kind": kind, **_draw_graph(rng, 20000, top)}


# ---- inputs ----


def _rng(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 1)
    return g


def _pairs_er(n, k, rng, _):
    return (torch.randint(0, n, (k,), generator=rng, device=DEV), torch.randint(0, n, (k,), generator=rng, device=DEV))


def _pairs_chung_lu(n, k, rng, case):
    """End points by weight (i + 1)^(-1 / (gamma - 1)), scaled to sum 2m and capped at 50 000 and n - 1."""
    w = torch.arange(1, n + 1, device=DEV, dtype=torch.float64).pow(-1.0 / (case["gamma"] - 1.0))
    w = (w * (2.0 * case["m"] / w.sum())).clamp(max=float(min(50000, n - 1)))
    cdf = w.cumsum(0)
    ends = [torch.searchsorted(cdf, torch.rand(k, generator=rng, device=DEV, dtype=torch.float64) * cdf[-1])
            for _ in range(2)]
    return tuple(e.clamp(max=n - 1) for e in ends)


def _pairs_rmat(n, k, rng, _):
    """(a, b, c, d) = (0.57, 0.19, 0.19, 0.05), no noise, no permutation."""
    u = torch.zeros(k, dtype=torch.int64, device=DEV)
    v = torch.zeros_like(u)
    for _level in range(n.bit_length() - 1):
        r = torch.rand(k, generator=rng, device=DEV)
        u.mul_(2).add_((r >= 0.76).to(torch.int64))
        v.mul_(2).add_((((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).to(torch.int64))
    return u, v


_PAIRS = {"er": _pairs_er, "chung_lu": _pairs_chung_lu, "rmat": _pairs_rmat}


def _edges(case, rng):
    """Exactly m distinct pairs u < v as sorted keys u * n + v: pairs drawn until there are enough, the excess
    dropped at random."""
    n, m = case["n"], case["m"]
    if case["gen"] == "er" and n * (n - 1) // 2 < 20 * m and n <= 8192:  # dense: m of all pairs
        iu = torch.triu_indices(n, n, 1, device=DEV)
        pick = torch.randperm(iu.shape[1], generator=rng, device=DEV)[:m].sort().values
        return iu[0][pick] * n + iu[1][pick]
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    while keys.numel() < m:
        k = int((m - keys.numel()) * 1.08) + 1024
        u, v = _PAIRS[case["gen"]](n, k, rng, case)
        lo, hi = torch.minimum(u, v), torch.maximum(u, v)
        new = (lo * n + hi)[lo != hi]
        keys = torch.unique(torch.cat([keys, new]))
    if keys.numel() > m:
        keep = torch.ones(keys.numel(), dtype=torch.bool, device=DEV)
        keep[torch.randperm(keys.numel(), generator=rng, device=DEV)[:keys.numel() - m]] = False
        keys = keys[keep]
    return keys


def _csr(case, rng):
    """Device CSR (row_ptr, col_idx), int32, rows ascending."""
    n = case["n"]
    keys = _edges(case, rng)
    both = torch.cat([keys, keys % n * n + keys // n]).sort().values
    rows = torch.div(both, n, rounding_mode="floor")
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.bincount(rows, minlength=n).cumsum(0)
    return rp.to(torch.int32), (both - rows * n).to(torch.int32)


def _small_graphs(case, rng, chunk=400):
    """A batch as one concatenated host CSR with local ids: n uniform in [n_lo, n_hi], even graphs Erdos-Renyi
    of density uniform in [0.05, 0.5], odd ones Chung-Lu of exponent uniform in [2, 3] and mean degree uniform
    in [2, min(32, (n - 1) / 4)]."""
    G, N = case["graphs"], case["n_hi"]
    n = torch.randint(case["n_lo"], N + 1, (G,), generator=rng, device=DEV)
    u = torch.rand((G, 3), generator=rng, device=DEV)
    i = torch.arange(N, device=DEV)
    deg, cols = [], []
    for g0 in range(0, G, chunk):
        ng, ug = n[g0:g0 + chunk], u[g0:g0 + chunk]
        inside = i[None, :] < ng[:, None]
        mean = 2.0 + ug[:, 2] * ((ng - 1) / 4.0).clamp(max=32.0).sub(2.0).clamp(min=0.0)
        w = (i + 1.0)[None, :].pow(-1.0 / (1.0 + ug[:, 1:2])) * inside
        w = w * (mean * ng / w.sum(1))[:, None]
        p = w[:, :, None] * w[:, None, :] / w.sum(1)[:, None, None]
        er = (torch.arange(g0, g0 + len(ng), device=DEV) % 2 == 0)[:, None, None]
        p = torch.where(er, (0.05 + 0.45 * ug[:, 0])[:, None, None], p)
        a = torch.rand(p.shape, generator=rng, device=DEV) < p
        a &= (i[:, None] < i[None, :])[None] & inside[:, :, None] & inside[:, None, :]
        a |= a.transpose(1, 2).clone()
        deg.append(a.sum(2)[inside])
        cols.append(a.nonzero()[:, 2].to(torch.int32))
    nv = n.cpu().numpy().astype(np.int32)
    d = torch.cat(deg).cpu().numpy().astype(np.int64)
    voff = np.concatenate([[0], np.cumsum(nv.astype(np.int64) + 1)])
    start = np.concatenate([[0], np.cumsum(nv.astype(np.int64))])
    ends = np.concatenate([[0], np.cumsum(d)])
    eoff = ends[start]
    rp = np.zeros(voff[-1], np.int32)
    at = np.arange(len(d)) + np.repeat(np.arange(G), nv) + 1  # place of every row's end
    rp[at] = ends[1:] - np.repeat(eoff[:-1], nv)
    return nv, voff, eoff, rp, torch.cat(cols).cpu().numpy()


def _requests(case, seed):
    """Host CSRs of Chung-Lu requests, edges log-uniform, exponent uniform in [2.1, 2.5], n = max(64, m / 8); the
    sizes are the same for every seed, the graphs are not."""
    sizes = np.random.RandomState(case["graphs"])
    out = []
    for r in range(case["graphs"]):
        m = int(round(math.exp(sizes.uniform(math.log(case["m_lo"]), math.log(case["m_hi"])))))
        c = {"gen": "chung_lu", "n": max(64, m // 8), "m": m, "gamma": float(sizes.uniform(2.1, 2.5))}
        rp, ci = _csr(c, _rng(seed * 1009 + r))
        out.append((rp.cpu().numpy(), ci.cpu().numpy()))
    return out


class _Batch:
    """A batch handle that is destroyed with its state."""

    def __init__(self, budget, flags):
        self.handle = gc.gc_batch_create(budget, flags)

    def __del__(self):
        gc.gc_batch_destroy(self.handle)


def prepare(case, seed):
    kind, rng = case["kind"], _rng(seed)
    state = {"kind": kind}
    if kind == "batch":
        state["graphs"] = _small_graphs(case, rng)
        state["batch"] = _Batch(64 << 30, gc.GC_BATCH_MANUAL)
    elif kind == "serve":
        state["graphs"] = _requests(case, seed)
        state["batch"] = _Batch(120 << 30, 0)
    else:
        rp, ci = _csr(case, rng)
        m = case["m"]
        if kind == "triangles":
            state.update(rp=rp, ci=ci, out=torch.empty(2 * m, dtype=torch.int32, device=DEV))
        elif kind == "whole":
            state.update(rp=rp.cpu().pin_memory(), ci=ci.cpu().pin_memory(),
                         rows=torch.empty((m, gc.GC_EDGE_COLS), dtype=torch.int64, pin_memory=True))
        else:
            stream = torch.cuda.current_stream()
            state["graph"] = gc.Graph(rp.cpu().numpy(), ci.cpu().numpy(), stream=stream)
            state["rows"] = torch.empty((m, gc.GC_EDGE_COLS), dtype=torch.int64, device=DEV)
            if kind == "induced":
                state["induced"] = torch.empty((m, gc.GC_INDUCED_COLS), dtype=torch.int64, device=DEV)
    return state


def _words(X):
    """128-bit counts as (low, high) words."""
    return np.array([[x & 0xffffffffffffffff, x >> 64] for x in X], np.uint64)


def run(state):
    kind = state["kind"]
    if kind == "count":
        X = state["graph"].count(state["rows"])
        return {"X": _words(X), "rows": state["rows"]}
    if kind == "induced":
        X = state["graph"].count_induced(state["induced"], state["rows"])
        return {"X": _words(X), "rows": state["rows"], "induced": state["induced"]}
    if kind == "whole":
        with gc.Graph(state["rp"], state["ci"], stream=torch.cuda.current_stream()) as g:
            X = g.count(state["rows"])
        return {"X": _words(X), "rows": state["rows"]}
    if kind == "batch":
        b = state["batch"].handle
        tickets = gc.gc_batch_submit_many(b, *state["graphs"])
        gc.gc_batch_flush(b)
        return {"X": gc.gc_batch_poll_many(b, tickets)}
    if kind == "serve":
        b = state["batch"].handle
        tickets = [gc.gc_batch_submit(b, rp, ci) for rp, ci in state["graphs"]]
        return {"X": gc.gc_batch_poll_many(b, tickets)}
    gc.gc_edge_triangles_noalloc(state["rp"], state["ci"], state["out"], stream=torch.cuda.current_stream())
    return {"triangles": state["out"]}


def work(case):
    """The bytes of one pass: the graph's CSR read once, every output written once. The counting itself is integer
    work on the chip (no floating-point operations)."""
    kind = case["kind"]
    if kind == "batch":
        n = np.arange(case["n_lo"], case["n_hi"] + 1, dtype=np.float64)
        mean = 2.0 + 0.5 * np.maximum(np.minimum(32.0, (n - 1) / 4) - 2.0, 0.0)
        nnz = np.mean(0.5 * 0.275 * n * (n - 1) + 0.5 * 0.95 * n * mean)
        return {"bytes": case["graphs"] * (4 * (nnz + n.mean() + 1) + 16 * gc.GC_NUM_GRAPHLETS), "flops": 0}
    if kind == "serve":
        lo, hi = case["m_lo"], case["m_hi"]
        m = (hi - lo) / math.log(hi / lo)
        return {"bytes": case["graphs"] * (4 * (2 * m + m / 8 + 1) + 16 * gc.GC_NUM_GRAPHLETS), "flops": 0}
    n, m = case["n"], case["m"]
    read = 4 * (2 * m + n + 1)
    if kind == "triangles":
        return {"bytes": read + 4 * 2 * m, "flops": 0}
    cols = gc.GC_EDGE_COLS + (gc.GC_INDUCED_COLS if kind == "induced" else 0)
    return {"bytes": read + 8 * cols * m + 16 * gc.GC_NUM_GRAPHLETS, "flops": 0}


# ---- the same counts by dense matrices ----


def _comb(x, k):
    r = 1
    for j in range(k):
        r = r * (x - j)
    return r // math.factorial(k) if x >= k else 0


def _dense_rows(A):
    """The 13 columns of every edge of the 0/1 matrix A (float64), by the definitions: T, S_u and S_v of each edge
    as 0/1 vectors, 4-cliques and induced 4-cycles as quadratic forms."""
    n = A.shape[0]
    deg = A.sum(1)
    m = int(deg.sum()) // 2
    out = []
    for u in range(n):
        vs = A[u, u + 1:].nonzero()[:, 0] + u + 1
        if not len(vs):
            continue
        au, av = A[u][None, :], A[vs]
        T = au * av
        Su, Sv = au - T, av - T
        Su[torch.arange(len(vs)), vs] = 0.0
        Sv[:, u] = 0.0
        t, su, sv = T.sum(1), Su.sum(1), Sv.sum(1)
        x7 = ((T @ A) * T).sum(1) / 2
        x10 = ((Su @ A) * Sv).sum(1)
        s, D = su + sv, n - 2 - t - su - sv
        out.append(torch.stack([t, s, D, x7, x10, t * (t - 1) / 2, t * s, su * (su - 1) / 2 + sv * (sv - 1) / 2,
                                su * sv, t * D, m - deg[u] - deg[vs] + 1, s * D, D * (D - 1) / 2], 1))
    if not out:
        return torch.zeros((0, 13), dtype=torch.int64, device=DEV)
    return torch.cat(out).round().to(torch.int64)


def _globals(rows, n, m):
    """X_1 .. X_17 from the summed columns (Sec. 4.6 of the paper)."""
    s = [int(x) for x in rows.sum(0)]
    C = dict(zip((3, 4, 5, 7, 10, 8, 9, 11, 12, 13, 14, 15, 16), s))
    X = {1: m, 2: _comb(n, 2) - m, 3: C[3] // 3, 4: C[4] // 2, 5: C[5]}
    X[6] = _comb(n, 3) - X[3] - X[4] - X[5]
    X[7] = C[7] // 6
    X[8] = C[8] - C[7]
    X[9] = (C[9] - 4 * X[8]) // 2
    X[10] = C[10] // 4
    X[11] = (C[11] - X[9]) // 3
    X[12] = C[12] - C[10]
    X[13] = (C[13] - X[9]) // 3
    X[14] = (C[14] - 6 * X[7] - 4 * X[8] - 2 * X[9] - 4 * X[10] - 2 * X[12]) // 2
    X[15] = (C[15] - 2 * X[12]) // 2
    X[16] = C[16] - 2 * X[14]
    X[17] = _comb(n, 4) - sum(X[i] for i in range(7, 17))
    return [X[i] for i in range(1, 18)]


def _dense(rp, ci):
    rp, ci = torch.as_tensor(rp, device=DEV).long(), torch.as_tensor(ci, device=DEV).long()
    n = len(rp) - 1
    A = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    A[torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1]), ci] = 1.0
    return A


def _slot_triangles(rp, ci, step=1 << 25):
    """|T| of the edge of every CSR slot: each triangle met once, as a pair of higher neighbours of its vertex
    lowest in (degree, id) that are adjacent."""
    rp, ci = rp.long(), ci.long()
    n, nnz = len(rp) - 1, len(ci)
    deg = rp[1:] - rp[:-1]
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    key = rows * n + ci
    rank = torch.empty(n, dtype=torch.int64, device=DEV)
    rank[torch.argsort(deg, stable=True)] = torch.arange(n, device=DEV)
    up = (rank[ci] > rank[rows]).nonzero()[:, 0]  # slots (a, b), a < b in rank
    first = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    first[1:] = torch.bincount(rows[up], minlength=n).cumsum(0)
    later = first[rows[up] + 1] - torch.arange(len(up), device=DEV) - 1  # out-slots of a after this one
    ends = later.cumsum(0)
    tri = torch.zeros(nnz, dtype=torch.int64, device=DEV)
    at = 0
    while at < len(up):
        base = int(ends[at - 1]) if at else 0
        to = max(at + 1, int(torch.searchsorted(ends, base + step)))
        cnt = later[at:to]
        i = torch.repeat_interleave(torch.arange(at, min(to, len(up)), device=DEV), cnt)
        j = i + 1 + torch.arange(len(i), device=DEV) - torch.repeat_interleave(ends[at:to] - cnt - base, cnt)
        b, c = ci[up[i]], ci[up[j]]
        pos = torch.searchsorted(key, b * n + c).clamp(max=nnz - 1)
        hit = key[pos] == b * n + c
        for s in (up[i][hit], up[j][hit], pos[hit]):
            tri += torch.bincount(s, minlength=nnz)
        at = to
    return (tri + tri[torch.searchsorted(key, ci * n + rows)]).to(torch.int32)


def exact(case, seed):
    """Whole numbers throughout: the counts themselves, for graphs small enough for dense matrices."""
    kind, rng = case["kind"], _rng(seed)
    if kind == "triangles":
        return {"triangles": _slot_triangles(*_csr(case, rng))}
    if kind == "batch" and case["graphs"] <= 64:
        nv, voff, eoff, rp, ci = _small_graphs(case, rng)
        X = []
        for g in range(case["graphs"]):
            A = _dense(rp[voff[g]:voff[g + 1]], ci[eoff[g]:eoff[g + 1]])
            X.append(_words(_globals(_dense_rows(A), int(nv[g]), int(eoff[g + 1] - eoff[g]) // 2)))
        return {"X": np.stack(X)}
    if kind in ("count", "whole") and case["n"] <= 4096:
        rows = _dense_rows(_dense(*_csr(case, rng)))
        return {"X": _words(_globals(rows, case["n"], case["m"])), "rows": rows}
    return None
