// gc_count.cu -- the triangle and 4-cycle passes, the per-edge finish and the
// derivation of the global counts.
//
// Work unit of pass C: one "v-group" = a vertex v and every edge e = (u, v)
// for which v is the high endpoint (P3, Sec. 4.3: d_v >= d_u, ties to the
// larger id). One CTA owns one unit at a time and a count table indexed by
// vertex; CTAs take units from an atomic cursor over the difficulty-ordered
// unit list (work stealing over Pi, Sec. 4.4).
//
// Pass T (gc_clique.cu) -- triangle step (Alg. 1): |T| per edge.
//
// Pass C -- 4-cycle step (Alg. 4/6) reorganised: P(e), the number of
//   4-cycles (as subgraphs) through e = #{(w, r) : w in Gamma(u)\{v},
//   r in Gamma(v)\{u}, w != r, w ~ r}, for all edges at once by counting
//   wedges from the highest-rank vertex of each cycle (see k_pass_c).
//
// Pass K (gc_clique.cu) -- 4-cliques x7 (Alg. 3/5) and
//   cross(e) = sum_{w in T} (|T_(w,u)| + |T_(w,v)| - 2) per edge.
//
// Finish -- per edge, Alg. 4/6's count #{(w, r) : w in S_u, r in S_v, w ~ r}:
//   for w in S_u, |Gamma(w) ∩ S_v| = |Gamma(w) ∩ Gamma(v)| - 1 - |Gamma(w) ∩ T|,
//   and sum_{w in S_u} |Gamma(w) ∩ T| = sum_{a in T} (|T_(a,u)| - 1) - 2 x7, so
//     x10 = P(e) - cross(e) + 2 x7.
//   Then the per-edge columns (Sec. 4.5) are written and the unrestricted
//   counts C_3..C_16 summed in 128 bits (per warp, then global atomics: local
//   aggregation communicated once, Sec. 4.6).
//
// Derive -- X_1..X_17 from the sums (Sec. 4.6, with X_11 = (C_11 - X_9)/3 and
//   C_9 = sum |T|(|S_u| + |S_v|)), exact 128-bit division checked.
#include <cuda_runtime.h>

#include <cstdlib>

#include "gc_deal.h"
#include "gc_internal.h"

namespace gc {
namespace {

__device__ __forceinline__ void atomic_add_u128(unsigned long long* p, u128 v) {
  unsigned long long lo = (unsigned long long)v;
  unsigned long long hi = (unsigned long long)(v >> 64);
  unsigned long long old = atomicAdd(p, lo);
  if (old + lo < old) hi += 1ull;
  if (hi) atomicAdd(p + 1, hi);
}

// Per-edge columns (Sec. 4.5): T, S_u, S_v of Fig. 2 and D_e.
__device__ __forceinline__ uint64_t edge_column(int k, int64_t t, int64_t su, int64_t sv, int64_t D,
                                                int64_t x7, int64_t x10, int64_t m_g, int64_t du,
                                                int64_t dv) {
  const int64_t s = su + sv;
  switch (k) {
    case 0: return (uint64_t)t;
    case 1: return (uint64_t)s;
    case 2: return (uint64_t)D;
    case 3: return (uint64_t)x7;
    case 4: return (uint64_t)x10;
    case 5: return (uint64_t)(t * (t - 1) / 2);
    case 6: return (uint64_t)(t * s);
    case 7: return (uint64_t)(su * (su - 1) / 2 + sv * (sv - 1) / 2);
    case 8: return (uint64_t)(su * sv);
    case 9: return (uint64_t)(t * D);
    case 10: return (uint64_t)(m_g - du - dv + 1);
    case 11: return (uint64_t)(s * D);
    default: return (uint64_t)(D * (D - 1) / 2);
  }
}

// Unrestricted count k (C_3 C_4 C_5 C_7 C_8 C_9 C_10 C_11 .. C_16) <- column
__device__ __forceinline__ int csum_column(int k) {
  // C_7 <- x7 (col 3), C_8 <- col 5, C_9 <- col 6, C_10 <- x10 (col 4)
  return k == 4 ? 5 : (k == 5 ? 6 : (k == 6 ? 4 : k));
}

template <bool kSmemTable>
__device__ __forceinline__ uint32_t* table_of(const DevGraph& g, const CountArgs& a, uint32_t* smem) {
  return kSmemTable ? smem : a.tables + (size_t)blockIdx.x * (size_t)g.table_n;
}

// ---------------- finish: x10, per-edge columns, sums ----------------
// One warp per 32 consecutive edges. Each lane computes the 13 columns of its
// edge into shared memory, and lane k < 13 adds column csum_column(k) of every
// row to its 128-bit running sum, flushed whenever the graph changes.
// kByEdge: the warp's edges are 32 consecutive edge ids, whose rows leave as
// one contiguous block of 416 words (13 coalesced stores of the warp) -- the
// order for rows written over the host link into pinned host memory.
// Otherwise: 32 consecutive out-slots (coalesced reads of the pass results),
// whose rows leave one at a time (13 lanes, one 104-byte store) -- the order
// for rows in device memory.
constexpr int kFinBlock = 256;
template <bool kByEdge>
__global__ void __launch_bounds__(kFinBlock) k_finish(DevGraph g, CountArgs a) {
  __shared__ unsigned long long st[kFinBlock / 32][32][13];
  __shared__ int32_t s_g[kFinBlock / 32];
  __shared__ long long s_edges[kFinBlock / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long(*rowv)[13] = st[warp];
  const unsigned long long* flat = &st[warp][0][0];
  u128 acc = 0;
  int32_t cur_g = -1;
  long long w_edges = 0;
  const int64_t stride = (int64_t)gridDim.x * (kFinBlock / 32) * 32;
  for (int64_t e0 = ((int64_t)blockIdx.x * (kFinBlock / 32) + warp) * 32; e0 < g.m; e0 += stride) {
    const int64_t i0 = e0 + lane;  // edge id (kByEdge) or out-slot
    int32_t gid = 0, eid = 0;
    if (i0 < g.m) {
      int32_t o = kByEdge ? g.e2o[i0] : (int32_t)i0;
      if ((uint32_t)o >= (uint32_t)g.m) o = 0;  // only for invalid input
      const int32_t p = g.ocsr[o];
      if (!kByEdge && a.per_edge) eid = g.eid[p];
      const int32_t r = g.rev[p];
      const int32_t u = g.ci[r], v = g.ci[p];
      gid = g.vgid ? g.vgid[u] : 0;
      const int64_t du = g.deg[u], dv = g.deg[v];
      const int64_t t = a.trio[o];
      const ulonglong2 xc = *reinterpret_cast<const ulonglong2*>(a.xc + 2 * (size_t)o);
      const int64_t x7 = a.x7d ? (int64_t)a.x7d[(size_t)u * g.n + v] : (int64_t)xc.x;
      const int64_t x10 = (int64_t)(a.P[p] + a.P[r]) - (int64_t)xc.y + 2 * x7;
      const int64_t su = du - t - 1, sv = dv - t - 1;
      const int64_t n_g = g.gn[gid], m_g = g.gm[gid];
      const int64_t D = n_g - 2 - t - su - sv;
#pragma unroll
      for (int c = 0; c < 13; ++c) rowv[lane][c] = edge_column(c, t, su, sv, D, x7, x10, m_g, du, dv);
    }
    __syncwarp();
    const int rows = (int)min((int64_t)32, (int64_t)g.m - e0);
    if (kByEdge && a.per_edge) {
      unsigned long long* dst = reinterpret_cast<unsigned long long*>(a.per_edge) + (size_t)e0 * 13;
      for (int i = lane; i < rows * 13; i += 32) dst[i] = flat[i];
    }
    for (int r = 0; r < rows; ++r) {
      const int32_t gr = __shfl_sync(0xffffffffu, gid, r);
      const int32_t er = __shfl_sync(0xffffffffu, eid, r);
      if (lane < 13) {
        if (!kByEdge && a.per_edge) a.per_edge[(size_t)er * 13 + lane] = rowv[r][lane];
        if (gr != cur_g) {
          if (cur_g >= 0) atomic_add_u128(a.csum + ((size_t)cur_g * 13 + lane) * 2, acc);
          acc = 0;
          cur_g = gr;
        }
        acc += (u128)rowv[r][csum_column(lane)];
      }
    }
    w_edges += rows;
    __syncwarp();
  }
  // the warps' last sums meet in shared memory: one atomic a block and column
  // where they belong to one graph (per warp, a count of ER-2000 sent 16 000
  // atomics to 26 words, 10 of the kernel's 16 us)
  __syncwarp();
  unsigned long long* fin = &st[warp][0][0];  // 13 low words, 13 high words
  if (lane < 13) {
    fin[lane] = (unsigned long long)acc;
    fin[13 + lane] = (unsigned long long)(acc >> 64);
  }
  if (lane == 0) {
    s_g[warp] = cur_g;
    s_edges[warp] = w_edges;
  }
  __syncthreads();
  if (threadIdx.x < 13) {
    u128 sum = 0;
    int32_t of = -1;
    for (int w = 0; w < kFinBlock / 32; ++w) {
      if (s_g[w] < 0) continue;
      if (s_g[w] != of) {
        if (of >= 0) atomic_add_u128(a.csum + ((size_t)of * 13 + threadIdx.x) * 2, sum);
        sum = 0;
        of = s_g[w];
      }
      const unsigned long long* f = &st[w][0][0];
      sum += ((u128)f[13 + threadIdx.x] << 64) | (u128)f[threadIdx.x];
    }
    if (of >= 0) atomic_add_u128(a.csum + ((size_t)of * 13 + threadIdx.x) * 2, sum);
  } else if (threadIdx.x == 13) {
    long long edges = 0;
    for (int w = 0; w < kFinBlock / 32; ++w) edges += s_edges[w];
    if (edges) atomicAdd(a.work + kWorkFinishEdges, (unsigned long long)edges);
  }
}

// ---------------- per-edge induced 4-node counts ----------------
// Per vertex x: vsum[2x] = sum over Gamma(x) of |T| of the edge (twice the
// triangles at x), vsum[2x + 1] = sum over Gamma(x) of the neighbour's
// degree. One warp per vertex, but a CTA per vertex for the g.n_long last ones, of
// more than 4096 neighbours each: a row's chains of loads (neighbour, degree; edge,
// out-slot, |T|) take 0.2 us per 32 entries of a warp, and the longest row was the
// kernel (a star of 100 000 leaves: 641 us, now 72).
constexpr int kLongRowBlock = 1024;
__global__ void __launch_bounds__(kLongRowBlock) k_vertex_sums_long(DevGraph g, const int32_t* __restrict__ trio,
                                                                    unsigned long long* __restrict__ vsum) {
  __shared__ unsigned long long s_sum[2][kLongRowBlock / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t x = g.n - 1 - (int32_t)blockIdx.x;
  const int32_t b = g.rp[x], d = g.rp[x + 1] - b;
  unsigned long long t2 = 0, ns = 0;
  for (int64_t k = threadIdx.x; k < d; k += kLongRowBlock) {
    ns += (unsigned long long)g.deg[g.ci[b + k]];
    t2 += (unsigned long long)trio[g.e2o[g.eid[b + k]]];
  }
  for (int o = 16; o; o >>= 1) {
    t2 += __shfl_xor_sync(0xffffffffu, t2, o);
    ns += __shfl_xor_sync(0xffffffffu, ns, o);
  }
  if (lane == 0) {
    s_sum[0][warp] = t2;
    s_sum[1][warp] = ns;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    unsigned long long v = 0;
    for (int w = 0; w < kLongRowBlock / 32; ++w) v += s_sum[threadIdx.x][w];
    vsum[2 * (size_t)x + threadIdx.x] = v;
  }
}
__global__ void __launch_bounds__(256) k_vertex_sums(DevGraph g, const int32_t* __restrict__ trio,
                                                     unsigned long long* __restrict__ vsum) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5), n = g.n - g.n_long;
  for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < n; x += warps) {
    unsigned long long t2 = 0, ns = 0;
    for (int32_t p = g.rp[x] + lane; p < g.rp[x + 1]; p += 32) {
      ns += (unsigned long long)g.deg[g.ci[p]];
      t2 += (unsigned long long)trio[g.e2o[g.eid[p]]];
    }
    for (int o = 16; o; o >>= 1) {
      t2 += __shfl_xor_sync(0xffffffffu, t2, o);
      ns += __shfl_xor_sync(0xffffffffu, ns, o);
    }
    if (lane == 0) {
      vsum[2 * x] = t2;
      vsum[2 * x + 1] = ns;
    }
  }
}

// For the edge e = (u, v) and the other vertices split into T, S_u, S_v (Fig.
// 2) and the rest R (|R| = D_e), the induced subgraph on {u, v, a, b} depends
// on the classes of a and b and on whether a ~ b. With A_XY the adjacent
// pairs between classes X and Y, the counts of H_7..H_16 containing e are
//   H7 = A_TT = x7            H8 = C(|T|,2) - A_TT + A_TS
//   H9 = |T||S| - A_TS + A_TR + A_SS                 H10 = A_SuSv = x10
//   H11 = C(|S_u|,2) + C(|S_v|,2) - A_SS             H12 = |S_u||S_v| - x10 + A_SR
//   H13 = |T||R| - A_TR      H14 = A_RR     H15 = |S||R| - A_SR     H16 = C(|R|,2) - A_RR
// (S = S_u + S_v, A_SS = A_SuSu + A_SvSv). The A's follow from quantities the
// passes already have, by counting incidences:
//   A_TS = cross(e) - 4 x7          (sum over T of |T_(w,u)| - 1 is 2 x7 + A_TSu)
//   A_SS = tri(u) + tri(v) - 2|T| - 2 x7 - A_TS      (triangles at u: |T| + x7 + A_TSu + A_SuSu)
//   A_TR = sum_T d_w - 2|T| - 2 x7 - A_TS            (degrees of T: u, v, T, S, R)
//   A_SR = sum_S d_w - |S| - A_TS - 2 A_SS - 2 x10   (sum_S d_w = NS(u) - d_v + NS(v) - d_u - 2 sum_T d_w)
//   A_RR = m - 1 - 2|T| - |S| - x7 - A_TS - A_SS - x10 - A_TR - A_SR
// with tri(x) the triangles at x and NS(x) the sum of the neighbours' degrees.
// Rows are staged per warp like k_finish (kByEdge: 32 consecutive edge ids).
constexpr int kIndCols = 10;
static_assert(kIndCols == GC_INDUCED_COLS, "induced columns");
template <bool kByEdge>
__global__ void __launch_bounds__(kFinBlock) k_finish_induced(DevGraph g, CountArgs a,
                                                              const unsigned long long* __restrict__ vsum,
                                                              unsigned long long* __restrict__ out) {
  __shared__ unsigned long long st[kFinBlock / 32][32][kIndCols];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long(*rowv)[kIndCols] = st[warp];
  const unsigned long long* flat = &st[warp][0][0];
  const int64_t stride = (int64_t)gridDim.x * (kFinBlock / 32) * 32;
  for (int64_t e0 = ((int64_t)blockIdx.x * (kFinBlock / 32) + warp) * 32; e0 < g.m; e0 += stride) {
    const int64_t i0 = e0 + lane;  // edge id (kByEdge) or out-slot
    int32_t eid = 0;
    if (i0 < g.m) {
      int32_t o = kByEdge ? g.e2o[i0] : (int32_t)i0;
      if ((uint32_t)o >= (uint32_t)g.m) o = 0;  // only for invalid input
      const int32_t p = g.ocsr[o];
      if (!kByEdge) eid = g.eid[p];
      const int32_t r = g.rev[p];
      const int32_t u = g.ci[r], v = g.ci[p];
      const int32_t gid = g.vgid ? g.vgid[u] : 0;
      const int64_t du = g.deg[u], dv = g.deg[v];
      const int64_t t = a.trio[o];
      const int64_t x7 = (int64_t)a.xc[2 * (size_t)o], cross = (int64_t)a.xc[2 * (size_t)o + 1];
      const int64_t x10 = (int64_t)(a.P[p] + a.P[r]) - cross + 2 * x7;
      const int64_t su = du - t - 1, sv = dv - t - 1, S = su + sv;
      const int64_t R = (int64_t)g.gn[gid] - 2 - t - S;
      const int64_t sdT = (int64_t)a.dsum[o];
      const int64_t aTS = cross - 4 * x7;
      const int64_t aSS = (int64_t)((vsum[2 * (size_t)u] + vsum[2 * (size_t)v]) / 2) - 2 * t - 2 * x7 - aTS;
      const int64_t aTR = sdT - 2 * t - 2 * x7 - aTS;
      const int64_t sdS = (int64_t)vsum[2 * (size_t)u + 1] - dv + (int64_t)vsum[2 * (size_t)v + 1] - du - 2 * sdT;
      const int64_t aSR = sdS - S - aTS - 2 * aSS - 2 * x10;
      const int64_t aRR = g.gm[gid] - 1 - 2 * t - S - x7 - aTS - aSS - x10 - aTR - aSR;
      unsigned long long* rw = rowv[lane];
      rw[0] = (unsigned long long)x7;
      rw[1] = (unsigned long long)(t * (t - 1) / 2 - x7 + aTS);
      rw[2] = (unsigned long long)(t * S - aTS + aTR + aSS);
      rw[3] = (unsigned long long)x10;
      rw[4] = (unsigned long long)(su * (su - 1) / 2 + sv * (sv - 1) / 2 - aSS);
      rw[5] = (unsigned long long)(su * sv - x10 + aSR);
      rw[6] = (unsigned long long)(t * R - aTR);
      rw[7] = (unsigned long long)aRR;
      rw[8] = (unsigned long long)(S * R - aSR);
      rw[9] = (unsigned long long)(R * (R - 1) / 2 - aRR);
    }
    __syncwarp();
    const int rows = (int)min((int64_t)32, (int64_t)g.m - e0);
    if (kByEdge) {
      unsigned long long* dst = out + (size_t)e0 * kIndCols;
      for (int i = lane; i < rows * kIndCols; i += 32) dst[i] = flat[i];
    } else {
      for (int r = 0; r < rows; ++r) {
        const int32_t er = __shfl_sync(0xffffffffu, eid, r);
        if (lane < kIndCols) out[(size_t)er * kIndCols + lane] = rowv[r][lane];
      }
    }
    __syncwarp();
  }
}

// ---------------- pass C: 4-cycles through every edge ----------------
// P(e) = number of 4-cycles (as subgraphs) containing e. Each 4-cycle is
// counted from its highest-rank vertex h: with cnt_h(o) = #{x in Gamma(h) :
// x < h, o in Gamma(x), o < h}, the wedge h-x-o closes cnt_h(o) - 1 cycles
// through h, each of which contains the edges (h, x) and (x, o) once. Ranks
// are the (degree, id) order of preprocessing P1/P3, so every wedge is met
// from one h only.
template <bool kSmemTable>
__global__ void __launch_bounds__(kBlock) k_pass_c(DevGraph g, CountArgs a) {
  extern __shared__ uint32_t smem[];
  __shared__ int32_t s_unit, s_next[3];
  uint32_t* tab = table_of<kSmemTable>(g, a, smem);
  const int lane = threadIdx.x & 31;
  const bool zero_all = kSmemTable && g.table_n <= 4096;
  long long w_wedge = 0;
  if (kSmemTable)
    for (int32_t i = threadIdx.x; i < g.table_n; i += kBlock) tab[i] = 0;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_unit = atomicAdd(a.cursor, 1);
    __syncthreads();
    const int32_t k = s_unit;
    if (k >= a.n_units) {
      if (lane == 0 && w_wedge) atomicAdd(a.work + kWorkCWedge, (unsigned long long)w_wedge);
      break;
    }
    const int32_t h = a.units[k];
    const int32_t base = g.gbase[g.vgid ? g.vgid[h] : 0];
    const int32_t hb = g.rp[h], he = g.rp[h + 1];
    if (threadIdx.x < 3) s_next[threadIdx.x] = hb;
    __syncthreads();
    // x runs over the lower-rank neighbours of h; o over those of x's
    // neighbours that rank below h (a prefix of Gamma(x): ids are ranks).
    for (int pass = 0; pass < (zero_all ? 2 : 3); ++pass) {
      for (;;) {
        int32_t p = 0;
        if (lane == 0) p = atomicAdd(&s_next[pass], 1);
        p = __shfl_sync(0xffffffffu, p, 0);
        if (p >= he) break;
        const int32_t x = g.ci[p];
        if (x >= h) break;  // the lower neighbours are a prefix of Gamma(h)
        const int32_t xb = g.rp[x];
        const int32_t xe = min(max(g.rev[p], xb), g.rp[x + 1]);  // Gamma(x) below the slot of (x, h) is < h
        unsigned long long s = 0;
        if (pass == 0 && lane == 0) w_wedge += xe - xb;
        for (int32_t q = xb + lane; q < xe; q += 32) {
          const int32_t o = g.ci[q];
          if (pass == 0) {
            atomicAdd(&tab[o - base], 1u);
          } else if (pass == 1) {
            const uint32_t c = tab[o - base] - 1u;
            if (c) {
              atomicAdd(&a.P[q], (unsigned long long)c);  // slot (x, o): consecutive over the lanes
              s += c;
            }
          } else {
            tab[o - base] = 0u;
          }
        }
        if (pass == 1) {
          for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (lane == 0 && s) atomicAdd(&a.P[p], s);  // slot (h, x)
        }
      }
      __syncthreads();
    }
    if (zero_all) {
      for (int32_t i = threadIdx.x; i < g.table_n; i += kBlock) tab[i] = 0;
    }
  }
}

// ---------------- graphs of at most kSmemTableMax vertices: rows of common neighbours ----------------
// For such a graph (of a union: every graph; which of them take this route:
// small_route) a row of counters c(w) = |Gamma(u)
// and Gamma(w)| over all vertices fits in shared memory, and gives for every
// edge (u, v)
//   |T|      = c(v)
//   P(e)     = sum over w in Gamma(v), w != u, of c(w) - 1
//   cross(e) = the sums over w in T of c(w) - 1 from u's row and from v's row
// in two sweeps over the rows of u's neighbours: one adds the counters, one,
// with a warp per neighbour v, reads them. So neither pass T nor pass C runs,
// and the 4-cliques (the rest of pass K) need nothing from here: both run side
// by side, where passes T and C, K, and the finish used to wait for each other
// (G(1000, 0.3): 480 -> 356 us per count; G(2000, 0.01): 123 -> 103 us). Work is
// sum d^2 counters, twice. CTA per vertex, largest degree first: in skewed graphs
// the largest one is the kernel (Chung-Lu 4000 / 60 000, 213 us: the SMs are busy
// 21 % of the time, and issue on 68 % of their active cycles).
constexpr int kRowBlock = 256;
constexpr uint32_t kMark = 0x80000000u;  // w is a neighbour of u
__global__ void __launch_bounds__(kRowBlock) k_rows(DevGraph g, CountArgs a) {
  extern __shared__ uint32_t cnt[];  // g.table_n
  __shared__ unsigned long long s_work;
  constexpr int kW = kRowBlock / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t u = g.n - 1 - (int32_t)blockIdx.x;
  const int32_t ub = g.rp[u], d = g.rp[u + 1] - ub;
  if (d == 0) return;
  const int32_t gid = g.vgid ? g.vgid[u] : 0;
  const int32_t base = g.gbase[gid], n = g.gn[gid];
  for (int32_t i = threadIdx.x; i < n; i += kRowBlock) cnt[i] = 0u;
  if (threadIdx.x == 0) s_work = 0ull;
  __syncthreads();
  // this warp's neighbours: warp, warp + kW, ..., 32 at a time, lane l the l-th
  for (int32_t i0 = warp; i0 < d; i0 += 32 * kW) {
    const int32_t i = i0 + kW * lane;
    int32_t xb = 0, xe = 0;
    if (i < d) {
      const int32_t x = g.ci[ub + i];
      xb = g.rp[x];
      xe = g.rp[x + 1];
      atomicOr(&cnt[x - base], kMark);
    }
    const int many = min(32, (d - i0 + kW - 1) / kW);
    for (int j = 0; j < many; ++j) {
      const int32_t b = __shfl_sync(0xffffffffu, xb, j), e = __shfl_sync(0xffffffffu, xe, j);
      for (int32_t q0 = b; q0 < e; q0 += 128) {  // four windows of loads in flight
        int32_t w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) w[t] = q0 + 32 * t + lane < e ? g.ci[q0 + 32 * t + lane] : -1;
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (w[t] >= 0) atomicAdd(&cnt[w[t] - base], 1u);
      }
    }
  }
  __syncthreads();
  long long w_read = 0;
  for (int32_t i0 = warp; i0 < d; i0 += 32 * kW) {
    const int32_t i = i0 + kW * lane;
    int32_t v = 0, vb = 0, ve = 0;
    if (i < d) {
      v = g.ci[ub + i];
      vb = g.rp[v];
      ve = g.rp[v + 1];
    }
    uint32_t my_p = 0, my_a = 0;
    const int many = min(32, (d - i0 + kW - 1) / kW);
    for (int j = 0; j < many; ++j) {
      const int32_t b = __shfl_sync(0xffffffffu, vb, j), e = __shfl_sync(0xffffffffu, ve, j);
      uint32_t p = 0, c = 0;  // below n^2 each
      for (int32_t q0 = b; q0 < e; q0 += 128) {
        int32_t w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) w[t] = q0 + 32 * t + lane < e ? g.ci[q0 + 32 * t + lane] : u;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const uint32_t x = w[t] == u ? 1u : cnt[w[t] - base];
          const uint32_t m = (x & ~kMark) - 1u;
          p += m;
          if (x & kMark) c += m;
        }
      }
      w_read += e - b;
      p = __reduce_add_sync(0xffffffffu, p);
      c = __reduce_add_sync(0xffffffffu, c);
      if (lane == j) {
        my_p = p;
        my_a = c;
      }
    }
    if (i < d) {
      // out-lists are the ends of the rows: the out-slot of the edge from the
      // slot of its lower end, p in row x, is out_ptr[x + 1] - (rp[x + 1] - p)
      const int32_t p = ub + i;
      const int32_t o = v > u ? g.out_ptr[u + 1] - (ub + d - p)
                              : g.out_ptr[v + 1] - (ve - min(max(g.rev[p], vb), ve - 1));
      if ((uint32_t)o < (uint32_t)g.m) {  // out of range only for invalid input
        if (v < u) {
          a.trio[o] = (int32_t)(cnt[v - base] & ~kMark);
          a.P[p] = my_p;
        }
        if (my_a) atomicAdd(&a.xc[2 * (size_t)o + 1], (unsigned long long)my_a);
      }
    }
  }
  if (lane == 0 && w_read) atomicAdd(&s_work, (unsigned long long)w_read);
  __syncthreads();
  if (threadIdx.x == 0) atomicAdd(a.work + kWorkCWedge, s_work);
}

// The same for a dense graph, on its bit rows. Row u's counters c(w), a lane
// per w, are kept as bit planes (a ballot per bit of c(w) - 1 and 32 vertices),
// so that the sums over Gamma(v), and over T = Gamma(u) and Gamma(v), of c(w) - 1
// are popcounts of row v, and of row v & row u, with each plane: a lane per v,
// words times bits operations for it where the lists took 25 instructions per
// 32 of its d_v entries. It waits on the loads of the bit rows, at 39 % of the warps
// an SM can hold (issue active 38 %, the pipe of popc 25 %). G(1000, 0.3): 165 -> 78 us.
constexpr int kDenseBits = 11;  // c(w) - 1 < 2^11
static_assert(kDenseMaxN <= 1 << kDenseBits, "counter planes");
constexpr int kRowDenseBlock = 128;
__global__ void __launch_bounds__(kRowDenseBlock, 8) k_rows_dense(DevGraph g, CountArgs a) {
  __shared__ uint32_t rowu[kDenseMaxN / 32];
  __shared__ __align__(16) uint32_t plane[kDenseMaxN / 32][12];
  __shared__ uint16_t cnt[kDenseMaxN];
  __shared__ unsigned long long s_work;
  constexpr int kW = kRowDenseBlock / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = g.n, W = (n + 31) / 32;
  const int32_t u = n - 1 - (int32_t)blockIdx.x;
  const int32_t ub = g.rp[u], d = g.rp[u + 1] - ub;
  if (d == 0) return;
  const int nb = 32 - __clz(d);  // c(w) <= d
  for (int i = threadIdx.x; i < W; i += kRowDenseBlock) rowu[i] = g.bits[(size_t)u * W + i];
  if (threadIdx.x == 0) s_work = 0ull;
  __syncthreads();
  for (int kb = warp; kb < W; kb += kW) {
    const int w = 32 * kb + lane;
    uint32_t c = 0;
    if (w < n) {
      const uint32_t* col = g.bits_t + w;
#pragma unroll 4
      for (int k = 0; k < W; ++k) c += __popc(col[(size_t)k * n] & rowu[k]);
      cnt[w] = (uint16_t)c;
    }
    const uint32_t x = w == u || c == 0u ? 0u : c - 1u;
    uint32_t mine = 0;
#pragma unroll
    for (int b = 0; b < kDenseBits; ++b) {
      const uint32_t p = __ballot_sync(0xffffffffu, (x >> b) & 1u);
      if (lane == b) mine = p;
    }
    if (lane < 12) plane[kb][lane] = mine;
  }
  __syncthreads();
  long long w_read = 0;
  for (int32_t i0 = 32 * warp; i0 < d; i0 += kRowDenseBlock) {
    const int32_t i = i0 + lane;
    const int32_t v = i < d ? g.ci[ub + i] : -1;
    const bool low = __any_sync(0xffffffffu, v >= 0 && v < u);  // the 4-cycles: from the higher end alone
    uint32_t pa[kDenseBits], pp[kDenseBits];
#pragma unroll
    for (int b = 0; b < kDenseBits; ++b) pa[b] = pp[b] = 0u;
    const uint32_t* col = g.bits_t + (v < 0 ? 0 : v);
    for (int k = 0; k < W; ++k) {
      const uint32_t x = v >= 0 ? col[(size_t)k * n] : 0u;
      const uint32_t y = x & rowu[k];
      const uint4* pl4 = reinterpret_cast<const uint4*>(plane[k]);
      const uint4 q0 = pl4[0], q1 = pl4[1], q2 = pl4[2];
      const uint32_t pl[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
#pragma unroll
      for (int b = 0; b < kDenseBits; ++b) {
        if (b < nb) {  // uniform
          pa[b] += __popc(y & pl[b]);
          if (low) pp[b] += __popc(x & pl[b]);
        }
      }
    }
    if (v < 0) continue;
    uint32_t sa = 0, sp = 0;
#pragma unroll
    for (int b = 0; b < kDenseBits; ++b) {
      sa += pa[b] << b;
      sp += pp[b] << b;
    }
    const int32_t vb = g.rp[v], ve = g.rp[v + 1], p = ub + i;
    w_read += ve - vb;
    const int32_t o = v > u ? g.out_ptr[u + 1] - (ub + d - p)
                            : g.out_ptr[v + 1] - (ve - min(max(g.rev[p], vb), ve - 1));
    if ((uint32_t)o < (uint32_t)g.m) {  // out of range only for invalid input
      if (v < u) {
        a.trio[o] = (int32_t)cnt[v];
        a.P[p] = sp;
      }
      if (sa) atomicAdd(&a.xc[2 * (size_t)o + 1], (unsigned long long)sa);
    }
  }
  if (w_read) atomicAdd(&s_work, (unsigned long long)w_read);
  __syncthreads();
  if (threadIdx.x == 0) atomicAdd(a.work + kWorkCWedge, s_work);
}

// 4-cliques of a dense graph by lowest vertex a: H_a on out(a) packed from the
// bit rows (a ballot per row and word), c_ij for its edges i < j, a lane each,
// added to x7d of the edge (b_i, b_j), and half of each member's sum to (a, b_i). No scan of out-lists, no hash and no list of edges, which
// took pass K's tiers 58 + 100 us on G(1000, 0.3); here 74 us. CTA per unit, largest
// first. Bound by instruction issue (72 % of the active cycles; popc's pipe 12 %).
constexpr int kDenseBlock = 256;
__host__ __device__ constexpr int dense_stride(int k) { return ((k + 31) / 32) | 1; }
__global__ void __launch_bounds__(kDenseBlock) k_cliques_dense(DevGraph g, CountArgs a, int32_t kmax) {
  extern __shared__ uint32_t hrow[];  // [kmax] rows, then the members and their sums
  int32_t* mem = reinterpret_cast<int32_t*>(hrow + (size_t)kmax * dense_stride(kmax));
  uint32_t* vx = reinterpret_cast<uint32_t*>(mem + kmax);
  __shared__ unsigned long long s_edges;
  __shared__ uint32_t s_queue[kDenseBlock / 32][64];
  constexpr int kW = kDenseBlock / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = g.n, Wn = (n + 31) / 32;
  const int32_t av = a.kunits[blockIdx.x], ob = g.out_ptr[av];
  const int k = min(g.out_ptr[av + 1] - ob, kmax);
  const int W = (k + 31) / 32, S = W | 1;
  for (int i = threadIdx.x; i < k; i += kDenseBlock) {
    mem[i] = g.out_idx[ob + i];
    vx[i] = 0u;
  }
  if (threadIdx.x == 0) s_edges = 0ull;
  __syncthreads();
  // pack: four rows of the graph at a time in registers (lane l words l and l +
  // 32), member j's bit from the lane that holds its word
  for (int i0 = 4 * warp; i0 < k; i0 += 4 * kW) {
    uint32_t lo[4], hi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const uint32_t* row = g.bits + (size_t)mem[min(i0 + t, k - 1)] * Wn;
      lo[t] = lane < Wn ? row[lane] : 0u;
      hi[t] = 32 + lane < Wn ? row[32 + lane] : 0u;
    }
    for (int b = 0; b < W; ++b) {
      const int j = 32 * b + lane;
      const int mj = j < k ? mem[j] : 0;
      const int sj = 31 - (mj & 31);
      uint32_t val = 0;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        uint32_t word = __shfl_sync(0xffffffffu, lo[t], (mj >> 5) & 31);
        if (Wn > 32) {  // uniform
          const uint32_t w2 = __shfl_sync(0xffffffffu, hi[t], (mj >> 5) & 31);
          if (mj >> 10) word = w2;
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, j < k && (int32_t)(word << sj) < 0);
        if (lane == t) val = bal;
      }
      if (lane < 4 && i0 + lane < k) hrow[(i0 + lane) * S + b] = val;
    }
  }
  __syncthreads();
  // the edges (i, j), i < j, of H_a go through a queue of the warp, so that a
  // lane takes one each (a lane per j of every row i, adjacent or not, read
  // three times as many words at density 0.3)
  uint32_t head = 0, tail = 0;
  uint32_t* queue = s_queue[warp];
  auto take = [&](uint32_t left) {
    if ((uint32_t)lane < left) {
      const uint32_t ij = queue[(head + lane) & 63u];
      const int i = (int)(ij >> 16), j = (int)(ij & 0xffffu);
      const uint32_t *hi = hrow + (size_t)i * S, *hj = hrow + (size_t)j * S;
      uint32_t c = 0;
#pragma unroll 4
      for (int w = 0; w < W; ++w) c += __popc(hi[w] & hj[w]);
      if (c) {
        atomicAdd(&a.x7d[(size_t)mem[i] * n + mem[j]], c);
        atomicAdd(&vx[i], c);
        atomicAdd(&vx[j], c);
      }
    }
    head += left;
    __syncwarp();
  };
  for (int b = 0; b < W; ++b) {
    const int last = min(32 * b + 31, k - 1);
    for (int i = warp; i < last; i += kW) {
      uint32_t on = hrow[(size_t)i * S + b];  // which j of the block are adjacent to i
      if (i >= 32 * b) on &= 0xffffffffu << ((i & 31) + 1);  // and above it (i < last: at most 31)
      if ((on >> lane) & 1u)
        queue[(tail + __popc(on & ((1u << lane) - 1u))) & 63u] = ((uint32_t)i << 16) | (uint32_t)(32 * b + lane);
      tail += __popc(on);
      __syncwarp();
      if (tail - head >= 32u) take(32u);
    }
  }
  const unsigned long long w_edges = tail;
  take(tail - head);
  if (lane == 0 && w_edges) atomicAdd(&s_edges, w_edges);
  __syncthreads();
  for (int i = threadIdx.x; i < k; i += kDenseBlock)
    if (vx[i]) atomicAdd(&a.x7d[(size_t)av * n + mem[i]], vx[i] >> 1);
  if (threadIdx.x == 0) {
    atomicAdd(a.work + kWorkKMembers, (unsigned long long)k);
    if (s_edges) {
      atomicAdd(a.work + kWorkKLocalEdges, s_edges);
      atomicAdd(a.work + kWorkTTriangles, s_edges);
      atomicAdd(a.work + kWorkKWords, s_edges * (unsigned long long)W);
    }
  }
}

// ---------------- pass C for hub units: the count table in shared memory ----------------
// The same wedges and attribution as k_pass_c, for the units h whose wedges
// (a few thousand hubs carry almost all of them on power-law graphs) would
// otherwise hit a vertex-indexed table in DRAM at random. Ids are ranks, so
// the lower-rank neighbours X of h are a prefix of Gamma(h) and, for x in X,
// the o < h are a prefix of Gamma(x), ascending. The o-range is swept in
// blocks of a.hub_tab words of shared-memory counters: cnt_h(o) for the block
// from each x's run of o in it, then the wedges of the block are attributed
// with the block's counts.
// Counter widths: cnt_h(o) <= d_o and ids ascend by degree, so the o-range has
// fixed segments of 2- to 32-bit counters (HubSeg), several to a block; o of
// degree 1 close no cycle and are skipped. On R-MAT scale 22 the id range of
// 4.2M takes 8 blocks and 12 segments where blocks of one 10-, 16- or 32-bit
// width took 31 to 94, so that a run has 72 entries instead of 16 (sweeps of
// (x, segment) 5.0e8, of (x, block) 2.2e9), and the segments' bounds in every longer row
// are looked up in a table made once per graph instead of searched. The
// whole kernel: 180 -> 127 ms there; 8.5 -> 5.6 ms on Chung-Lu 1M, where
// about a quarter of the warps' time is still the barrier between a block's
// two phases, and the shared-memory pipe, with three-way bank conflicts of
// random counters, is busy half of the time.
// In both phases a warp works on a chunk of up to 32 x's: for a hub of more
// than 1024 x's it takes chunks from a shared counter, heaviest first; for a
// smaller hub each warp keeps one chunk, x = w, w + 32, ..., so that the
// warps carry about equal work. run_chunk orders the loads of a chunk's runs
// so that consecutive lanes load, and add to, consecutive slots. The block
// fills shared memory up to the step of the L1 carveout that kHubTabDefault
// explains: the longer the runs per block, the fewer the sweeps.
constexpr int kHeavyBlock = 1024;
constexpr int kHeavyWarps = kHeavyBlock / 32;
constexpr int32_t kFine = 256;  // heaviest x's of a large hub, four to a chunk

// Counters of a segment, 2^lg to a word (no count of the segment reaches its
// field's size, so no carry crosses into the next field).
struct Fields {
  int lg;         // log2 of the counters per word
  int sh;         // log2 of a counter's bits
  uint32_t low;   // counters per word - 1
  uint32_t mask;  // a counter's bits
  __device__ __forceinline__ explicit Fields(int l)
      : lg(l), sh(5 - l), low((1u << l) - 1u), mask(l ? (1u << (32 >> l)) - 1u : 0xffffffffu) {}
};
__device__ __forceinline__ void add_count(uint32_t* tab, uint32_t slot, const Fields& f) {
  atomicAdd(&tab[slot >> f.lg], 1u << ((slot & f.low) << f.sh));
}
__device__ __forceinline__ uint32_t read_count(const uint32_t* tab, uint32_t slot, const Fields& f) {
  return (tab[slot >> f.lg] >> ((slot & f.low) << f.sh)) & f.mask;
}

// first index in [p, e) with a[index] >= key; a ascending
__device__ __forceinline__ int32_t gallop_lower_bound(const int32_t* __restrict__ a, int32_t p, int32_t e,
                                                      int32_t key) {
  if (p >= e || a[p] >= key) return p;
  int32_t lo = p, step = 1;  // a[lo] < key throughout; lo + step or lo + hi may pass 2^31
  while (step < e - lo && a[lo + step] < key) {
    lo += step;
    step <<= 1;
  }
  int32_t hi = step < e - lo ? lo + step : e;
  ++lo;
  while (lo < hi) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    if (a[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The runs of one chunk, in one segment: lane l's run is [st, st + L) of
// Gamma(x) for its x (L = 0 for none), all its o in the segment that starts at
// lo_id and whose counters start at tab. kAttr = false counts each o; true
// attributes each wedge: cnt_h(o) - 1 to the slot (x, o), and the sum over the
// run to `acc` of the run's lane (the slot (h, x)). Entries are loaded 32
// consecutive ones to a window, in three steps by what the run has left, so
// that no window is issued for nothing and several loads are in flight:
// whole blocks of eight windows, one run at a time; the other whole windows,
// of all runs end to end; and the last < 32 entries of every run, dealt to the
// lanes end to end. (One step of eight windows for any run of 32 entries or
// more, as before, left more than half of the windows of runs of about 100
// entries empty: 75 instructions per 32 wedges on R-MAT scale 18.) Sums over
// the distinct o of a run stay in 32 bits: cnt_h(o) <= d_o, and all degrees
// sum to 2m < 2^31.
template <bool kAttr>
__device__ __forceinline__ void run_chunk(const DevGraph& g, const CountArgs& a, uint32_t* tab, uint32_t* sx32,
                                          int32_t* comp, int32_t st, int32_t L, int32_t lo_id, const Fields& f,
                                          int lane, unsigned long long& acc) {
  // one window's entry o at slot q; returns its count for the sum
  auto one = [&](int32_t o, int32_t q) -> uint32_t {
    const uint32_t slot = (uint32_t)(o - lo_id);
    if (!kAttr) {
      add_count(tab, slot, f);
      return 0u;
    }
    const uint32_t cnt = read_count(tab, slot, f) - 1u;
    if (cnt) atomicAdd(&a.P[q], (unsigned long long)cnt);
    return cnt;
  };
  unsigned lm = __ballot_sync(0xffffffffu, L >= 256);
  while (lm) {
    const int src = __ffs(lm) - 1;
    lm &= lm - 1;
    const int32_t* s0 = g.ci + __shfl_sync(0xffffffffu, st, src);
    const int32_t n0 = __shfl_sync(0xffffffffu, L, src) & ~255;
    for (int32_t k = lane; k < n0; k += 256) {
      int32_t o[8];
      uint32_t sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = s0[k + 32 * j];
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += one(o[j], (int32_t)(s0 - g.ci) + k + 32 * j);
      if (kAttr) {
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == src) acc += sum;
      }
    }
  }
  // whole windows left: at most seven a run
  st += L & ~255;
  L &= 255;
  {
    int32_t incl = L >> 5;
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int32_t total = __shfl_sync(0xffffffffu, incl, 31);
    const int32_t base = st - 32 * (incl - (L >> 5));  // window w of this run starts at base + 32 w
    for (int32_t w0 = 0; w0 < total; w0 += 4) {
      int32_t q[4], o[4], own[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        own[j] = __popc(__ballot_sync(0xffffffffu, incl <= w0 + j)) & 31;  // & 31: past the last window
        q[j] = __shfl_sync(0xffffffffu, base, own[j]) + 32 * (w0 + j) + lane;
        o[j] = w0 + j < total ? g.ci[q[j]] : -1;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (w0 + j >= total) break;  // warp-uniform
        uint32_t cnt = one(o[j], q[j]);
        if (kAttr) {
          cnt = __reduce_add_sync(0xffffffffu, cnt);
          if (lane == own[j]) acc += cnt;
        }
      }
    }
  }
  // the last entries of every run, dealt to the lanes end to end
  st += L & ~31;
  L &= 31;
  if (kAttr) {
    sx32[lane] = 0u;
    __syncwarp();
  }
  const Deal d = deal_setup(L, comp, lane);
  const int32_t sb = st - d.excl;  // slot of position kk of this lane's run: sb + kk
  int before = 0;
  for (int32_t k0 = 0; k0 < d.total; k0 += 128) {
    int32_t q[4], ol[4], o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      ol[j] = deal_owner(d, L, k0 + 32 * j, comp, lane, before);
      const int32_t kk = k0 + 32 * j + lane;
      const int32_t bj = __shfl_sync(0xffffffffu, sb, ol[j]);
      q[j] = kk < d.total ? bj + kk : -1;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = q[j] >= 0 ? g.ci[q[j]] : lo_id;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (q[j] < 0) continue;
      const uint32_t cnt = one(o[j], q[j]);
      if (kAttr && cnt) atomicAdd(&sx32[ol[j]], cnt);  // the owner's sum
    }
  }
  __syncwarp();
  if (kAttr) {
    acc += sx32[lane];
    __syncwarp();
  }
}

// The run {o in Gamma(x) : o in the segment, in the job's o-range [jlo, jhi),
// o < h} of a lower neighbour x of h: [st, st + L). `k` is the segment's place
// in its graph; rend the slot of (x, h). Rows with a position table read the
// segment's bounds there; the others (at most max(31, segments) entries) are
// searched; a job that starts or ends inside the segment is searched too.
__device__ __forceinline__ void hub_run(const DevGraph& g, const HubGeom& ge, const HubSeg& sg, int32_t k, int32_t x,
                                        int32_t rend, int32_t jlo, int32_t jhi, int32_t& st, int32_t& L) {
  int32_t en;
  if (x >= ge.xmin) {
    const int32_t* pp = g.hpos + ge.pos + (int64_t)(x - ge.xmin) * (ge.nseg + 1) + k;
    st = pp[0];
    en = min(pp[1], rend);
    if (jlo > sg.lo) st = gallop_lower_bound(g.ci, st, en, jlo);
  } else {
    st = gallop_lower_bound(g.ci, g.rp[x], rend, max(jlo, sg.lo));
    en = gallop_lower_bound(g.ci, st, rend, sg.hi);
  }
  if (jhi < sg.hi) en = gallop_lower_bound(g.ci, st, en, jhi);
  L = max(en - st, 0);
}

__global__ void __launch_bounds__(kHeavyBlock, 1) k_pass_c_heavy(DevGraph g, CountArgs a) {
  extern __shared__ uint32_t tab[];  // a.hub_tab words of counters
  __shared__ int32_t s_unit, s_nx, s_chunk[2];
  const unsigned long long t_start = global_ns();
  __shared__ uint32_t s_sx32[kHeavyWarps][32];  // the short runs' part (< 32 entries x counts < 2^26)
  __shared__ int32_t s_comp[kHeavyWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int32_t* comp = s_comp[warp];
  long long w_wedge = 0, w_sweeps = 0, w_jobs = 0;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_unit = atomicAdd(a.cursor + 8, 1);
    __syncthreads();
    const int32_t jb = s_unit;
    if (jb >= a.n_cjobs) break;
    const int4 job = a.cjobs[jb];  // hub (index into cunits), its o-range [y, z), 2 x segment of y + first
    const int32_t h = a.cunits[job.x];
    const HubGeom ge = g.hgeom[g.vgid ? g.vgid[h] : 0];
    const int32_t hb = g.rp[h], he = g.rp[h + 1];
    if (threadIdx.x == 0) {
      int32_t lo = hb, hi = he;  // first slot of Gamma(h) with id >= h
      while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);  // slots beyond 2^30: their sum is no int32
        if (g.ci[mid] < h) lo = mid + 1; else hi = mid;
      }
      s_nx = lo - hb;
    }
    __syncthreads();
    const int32_t nx = s_nx;
    // chunks of x's: of consecutive ones, taken heaviest first (X ascends by
    // degree) from a shared counter, when there are more than a CTA's threads
    // -- four to a chunk for the heaviest, so that no warp keeps the others
    // waiting with 32 of them (pass C of Chung-Lu 1M 7.94 -> 7.54 ms), 32 to a
    // chunk for the rest; otherwise one chunk per warp, x = warp, warp + 32, ...
    const bool small = nx <= kHeavyBlock;
    const int32_t fine = min(nx, kFine), fine_chunks = (fine + 3) >> 2;
    const int32_t nchunks = small ? kHeavyWarps : fine_chunks + ((nx - fine + 31) >> 5);
    if (job.w & 1) {  // the hub's wedges, counted by its first job
      for (int32_t i = threadIdx.x; i < nx; i += kHeavyBlock) {
        const int32_t xb = g.rp[g.ci[hb + i]];
        w_wedge += max(g.rev[hb + i], xb) - xb;  // Gamma(x) below the slot of (x, h) is < h
      }
    }
    if (threadIdx.x == 0) ++w_jobs;
    const int32_t jlo = job.y, jhi = job.z, seg_end = ge.seg + ge.nseg;
    const int32_t jcut = jhi == h ? 0x7fffffff : jhi;  // runs end below h by themselves
    // this thread's x when its chunk is fixed
    int32_t rx = 0, rrend = 0;
    const int32_t ri = warp + kHeavyWarps * lane;
    if (small && ri < nx) {
      rx = g.ci[hb + ri];
      rrend = min(max(g.rev[hb + ri], g.rp[rx]), g.rp[rx + 1]);
    }
    for (int32_t s0 = job.w >> 1, s1; s0 < seg_end && g.hseg[s0].lo < jhi; s0 = s1) {
      // one block: segments [s0, s1)
      int32_t words = 0;
      const int32_t w0 = g.hseg[s0].word;
      for (s1 = s0; s1 < seg_end;) {
        const HubSeg sg = g.hseg[s1];
        if (sg.lo >= jhi) break;
        words = sg.word - w0 + ((min(sg.hi, jhi) - sg.lo + (1 << sg.lg) - 1) >> sg.lg);
        ++s1;
        if (sg.last) break;
      }
      for (int32_t i = threadIdx.x; i < words; i += kHeavyBlock) tab[i] = 0u;
      if (threadIdx.x == 0) {
        w_sweeps += (long long)nx * (s1 - s0);
        s_chunk[0] = 0;
        s_chunk[1] = 0;
      }
      __syncthreads();
      for (int phase = 0; phase < 2; ++phase) {  // the block's counts, then the attribution of its wedges
        for (int32_t c = 0;;) {
          if (!small) {
            if (lane == 0) c = atomicAdd(&s_chunk[phase], 1);
            c = __shfl_sync(0xffffffffu, c, 0);
            if (c >= nchunks) break;
          }
          int32_t i = ri;
          if (!small) {
            const bool few = c < fine_chunks;
            const int32_t k = few ? 4 * c + lane : fine + 32 * (c - fine_chunks) + lane;  // from the heaviest x down
            i = (few && (lane >= 4 || k >= fine)) || k >= nx ? nx : nx - 1 - k;
          }
          int32_t x = rx, rend = rrend;
          if (!small && i < nx) {
            x = g.ci[hb + i];
            rend = min(max(g.rev[hb + i], g.rp[x]), g.rp[x + 1]);
          }
          unsigned long long acc = 0;  // this x's wedges' counts
          for (int32_t s = s0; s < s1; ++s) {
            const HubSeg sg = g.hseg[s];
            const Fields f(sg.lg);
            int32_t st = 0, L = 0;
            if (i < nx) hub_run(g, ge, sg, s - ge.seg, x, rend, jlo, jcut, st, L);
            if (phase == 0)
              run_chunk<false>(g, a, tab + (sg.word - w0), s_sx32[warp], comp, st, L, sg.lo, f, lane, acc);
            else
              run_chunk<true>(g, a, tab + (sg.word - w0), s_sx32[warp], comp, st, L, sg.lo, f, lane, acc);
          }
          if (acc) atomicAdd(&a.P[hb + i], acc);  // slot (h, x); only runs of x in [0, nx) add to acc
          if (small) break;
        }
        __syncthreads();
      }
    }
  }
  for (int o = 16; o; o >>= 1) w_wedge += __shfl_xor_sync(0xffffffffu, w_wedge, o);
  if (lane == 0 && w_wedge) {
    atomicAdd(a.work + kWorkCWedge, (unsigned long long)w_wedge);
    atomicAdd(a.work + kWorkCHeavyWedge, (unsigned long long)w_wedge);
  }
  if (threadIdx.x == 0) {
    if (w_sweeps) atomicAdd(a.work + kWorkCBlocks, (unsigned long long)w_sweeps);
    if (w_jobs) atomicAdd(a.work + kWorkCHubJobs, (unsigned long long)w_jobs);
    const unsigned long long life = global_ns() - t_start;
    atomicAdd(a.work + kWorkCHubCtas, 1ull);
    atomicAdd(a.work + kWorkCHubBusySum, life);
    atomicMax(a.work + kWorkCHubBusyMax, life);
  }
}

// ---------------- pass C for units of at most kHashMaxW wedges ----------------
// The same wedges and attribution as k_pass_c, with cnt_h(o) in a
// shared-memory hash keyed by o instead of a vertex-indexed table in DRAM
// (open addressing, linear probing; sized per unit to at least twice its
// wedges, so at most half full; 16-bit counts, since cnt_h(o) <= wedges).
// A warp takes one lower neighbour x of h at a time, its lanes the run
// {o in Gamma(x) : o < h}, which ends at the slot of (x, h) (ids are ranks
// and rows ascend).
constexpr int kHashBlock = 512;
constexpr int kHashSmallBlock = 128;
constexpr int kHashMidBlock = 256;

__device__ __forceinline__ uint32_t o_hash(int32_t o, int bits) {
  return ((uint32_t)o * 0x9E3779B1u) >> (32 - bits);  // Fibonacci hashing
}
// slot of o (inserted if absent), or -1 if the table is full
__device__ __forceinline__ int32_t hash_insert(int32_t* keys, int32_t o, uint32_t mask, int bits) {
  uint32_t sl = o_hash(o, bits);
  for (uint32_t t = 0; t <= mask; ++t) {
    const int32_t kk = *reinterpret_cast<volatile int32_t*>(&keys[sl]);
    if (kk == o) return (int32_t)sl;
    if (kk == -1) {
      const int32_t prev = atomicCAS(&keys[sl], -1, o);
      if (prev == -1 || prev == o) return (int32_t)sl;
    }
    sl = (sl + 1) & mask;
  }
  return -1;
}
// slot of o, or -1 if absent
__device__ __forceinline__ int32_t hash_find(const int32_t* keys, int32_t o, uint32_t mask, int bits) {
  uint32_t sl = o_hash(o, bits);
  for (uint32_t t = 0; t <= mask; ++t) {
    const int32_t kk = keys[sl];
    if (kk == o) return (int32_t)sl;
    if (kk == -1) return -1;
    sl = (sl + 1) & mask;
  }
  return -1;
}

// Three instances: 512-thread CTAs, two an SM, with the table for kHashMaxW
// wedges; 256-thread CTAs, eight an SM, for units of at most kHashMidW; and,
// for the many units of at most kHashSmallW wedges (on R-MAT scale 22, 87 %
// of the hashed units and 10 % of their wedges), 128-thread CTAs with a table
// for kHashSmallW, sixteen an SM, so that a unit's barriers and latency
// chains no longer hold a large CTA. Units [k0, k1) of the hashed list
// (heaviest first), taken from *cursor.
template <int kThreads, int kMaxW>
__global__ void __launch_bounds__(kThreads, kThreads == kHashBlock ? kCtasPerSm : 2048 / kThreads)
    k_pass_c_hash(DevGraph g, CountArgs a, int32_t k0, int32_t k1, int32_t* cursor) {
  extern __shared__ int32_t hkeys[];                                  // [2 kMaxW] o, or -1
  uint32_t* hcnt = reinterpret_cast<uint32_t*>(hkeys + 2 * kMaxW);    // [kMaxW] two counts
  __shared__ int32_t s_unit, s_next[2];
  __shared__ unsigned long long s_wedge;
  if (threadIdx.x == 0) s_wedge = 0ull;  // seen by all after the loop's first barrier
  const int lane = threadIdx.x & 31;
  long long w_wedge = 0;  // lane 0
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_unit = k0 + atomicAdd(cursor, 1);
    __syncthreads();
    const int32_t k = s_unit;
    if (k >= k1) break;
    const int32_t h = a.cunits[a.n_cheavy + k];
    const int32_t wk = min(a.chash_w[k], (int32_t)kMaxW);
    int bits = 6;
    while ((1 << bits) < 2 * wk) ++bits;  // at most log2(2 * kHashMaxW)
    const uint32_t mask = (1u << bits) - 1u;
    const int32_t hb = g.rp[h], he = g.rp[h + 1];
    for (int32_t i = threadIdx.x; i <= (int32_t)mask; i += kThreads) hkeys[i] = -1;
    for (int32_t i = threadIdx.x; i <= (int32_t)(mask >> 1); i += kThreads) hcnt[i] = 0u;
    if (threadIdx.x < 2) s_next[threadIdx.x] = hb;
    __syncthreads();
    // pass 0 counts cnt_h(o); pass 1 attributes cnt_h(o) - 1 to the slots
    // (x, o) and, summed over the run, to (h, x)
    for (int pass = 0; pass < 2; ++pass) {
      for (;;) {
        int32_t p = 0;
        if (lane == 0) p = atomicAdd(&s_next[pass], 1);
        p = __shfl_sync(0xffffffffu, p, 0);
        if (p >= he) break;
        const int32_t x = g.ci[p];
        if (x >= h) break;  // the lower neighbours are a prefix of Gamma(h)
        const int32_t xb = g.rp[x];
        const int32_t xe = min(max(g.rev[p], xb), g.rp[x + 1]);  // Gamma(x) below the slot of (x, h)
        if (pass == 0 && lane == 0) w_wedge += xe - xb;
        uint32_t sx = 0u;
        for (int32_t q0 = xb; q0 < xe; q0 += 128) {  // four windows of 32 in flight
          int32_t o[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int32_t q = q0 + 32 * j + lane;
            o[j] = q < xe ? g.ci[q] : -1;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (o[j] < 0) continue;
            if (pass == 0) {
              const int32_t sl = hash_insert(hkeys, o[j], mask, bits);
              if (sl >= 0) atomicAdd(&hcnt[sl >> 1], 1u << ((sl & 1) << 4));
              else atomicOr(a.status, (int32_t)kSpillOverflow);  // more distinct o than wedges: invalid input
            } else {
              const int32_t sl = hash_find(hkeys, o[j], mask, bits);
              const uint32_t c = sl >= 0 ? ((hcnt[sl >> 1] >> ((sl & 1) << 4)) & 0xffffu) - 1u : 0u;
              if (c) {
                atomicAdd(&a.P[q0 + 32 * j + lane], (unsigned long long)c);  // slot (x, o)
                sx += c;
              }
            }
          }
        }
        if (pass == 1) {
          for (int off = 16; off; off >>= 1) sx += __shfl_xor_sync(0xffffffffu, sx, off);
          if (lane == 0 && sx) atomicAdd(&a.P[p], (unsigned long long)sx);  // slot (h, x)
        }
      }
      __syncthreads();
    }
  }
  if (lane == 0 && w_wedge) atomicAdd(&s_wedge, (unsigned long long)w_wedge);
  __syncthreads();
  if (threadIdx.x == 0 && s_wedge) {  // one atomic a block
    atomicAdd(a.work + kWorkCWedge, s_wedge);
    atomicAdd(a.work + kWorkCHashWedge, s_wedge);
  }
}

// ---------------- pass C for units of at most kHash2MaxW wedges ----------------
// The same counting and attribution as k_pass_c_hash, for the units whose
// wedges do not fit that hash: each slot is one 32-bit word holding the
// vertex o (22 bits, from its graph's first; graphs of at most 2^22 vertices) and cnt_h(o) (10 bits;
// units of fewer than 1023 lower neighbours, so a count never reaches 1023
// and a word is never all ones, the empty mark). kHash2Slots words fill the
// shared memory of one 1024-thread CTA per SM; a unit uses the first
// ceil(W / 0.72) of them, so the table is at most 72 % full, and the probe
// position is a multiply-shift of the hash into that range.
constexpr int kHash2Block = 1024;
constexpr uint32_t kHash2Empty = 0xffffffffu;

__device__ __forceinline__ uint32_t h2_start(int32_t o, uint32_t size) {
  return (uint32_t)(((unsigned long long)((uint32_t)o * 0x9E3779B1u) * size) >> 32);
}
// adds 1 to the count of o (inserted with count 1 if absent); false if the
// table is full (cannot happen for a unit sized as above)
__device__ __forceinline__ bool h2_insert(uint32_t* tab, int32_t o, uint32_t size) {
  uint32_t sl = h2_start(o, size);
  for (uint32_t t = 0; t < size; ++t) {
    uint32_t w = *reinterpret_cast<volatile uint32_t*>(&tab[sl]);
    if (w == kHash2Empty) {
      w = atomicCAS(&tab[sl], kHash2Empty, ((uint32_t)o << 10) | 1u);
      if (w == kHash2Empty) return true;
    }
    if ((w >> 10) == (uint32_t)o) {
      atomicAdd(&tab[sl], 1u);
      return true;
    }
    sl = sl + 1 == size ? 0 : sl + 1;
  }
  return false;
}
__device__ __forceinline__ uint32_t h2_count(const uint32_t* tab, int32_t o, uint32_t size) {
  uint32_t sl = h2_start(o, size);
  for (uint32_t t = 0; t < size; ++t) {
    const uint32_t w = tab[sl];
    if (w == kHash2Empty) return 0u;
    if ((w >> 10) == (uint32_t)o) return w & 1023u;
    sl = sl + 1 == size ? 0 : sl + 1;
  }
  return 0u;
}

// Two instances: 1024-thread CTAs with the whole table, one an SM; and
// 512-thread CTAs with half of it, two an SM, for the units of at most
// kHash2HalfMaxW wedges. Units [k0, k1) of the packed-key list (heaviest
// first), taken from *cursor.
template <int kThreads, int kSlots>
__global__ void __launch_bounds__(kThreads, kThreads == kHash2Block ? 1 : 2)
    k_pass_c_hash2(DevGraph g, CountArgs a, int32_t k0, int32_t k1, int32_t* cursor) {
  extern __shared__ uint32_t htab[];  // kSlots packed (o, count) words
  __shared__ int32_t s_unit, s_next[2];
  __shared__ unsigned long long s_wedge;
  if (threadIdx.x == 0) s_wedge = 0ull;  // seen by all after the loop's first barrier
  const int lane = threadIdx.x & 31;
  long long w_wedge = 0;  // lane 0
  const int32_t first = a.n_cheavy + a.n_chash;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_unit = k0 + atomicAdd(cursor, 1);
    __syncthreads();
    const int32_t k = s_unit;
    if (k >= k1) break;
    const int32_t h = a.cunits[first + k];
    const int32_t wk = min(a.chash_w[a.n_chash + k], (int32_t)kHash2MaxW);
    const int32_t base = g.gbase[g.vgid ? g.vgid[h] : 0];
    const uint32_t size = min((uint32_t)kSlots, (uint32_t)(((long long)wk * 25 + 17) / 18) + 32u);
    const int32_t hb = g.rp[h], he = g.rp[h + 1];
    for (uint32_t i = threadIdx.x; i < size; i += kThreads) htab[i] = kHash2Empty;
    if (threadIdx.x < 2) s_next[threadIdx.x] = hb;
    __syncthreads();
    // pass 0 counts cnt_h(o); pass 1 attributes cnt_h(o) - 1 to the slots
    // (x, o) and, summed over the run, to (h, x)
    for (int pass = 0; pass < 2; ++pass) {
      for (;;) {
        int32_t p = 0;
        if (lane == 0) p = atomicAdd(&s_next[pass], 1);
        p = __shfl_sync(0xffffffffu, p, 0);
        if (p >= he) break;
        const int32_t x = g.ci[p];
        if (x >= h) break;  // the lower neighbours are a prefix of Gamma(h)
        const int32_t xb = g.rp[x];
        const int32_t xe = min(max(g.rev[p], xb), g.rp[x + 1]);  // Gamma(x) below the slot of (x, h)
        if (pass == 0 && lane == 0) w_wedge += xe - xb;
        unsigned long long sx = 0;
        for (int32_t q0 = xb; q0 < xe; q0 += 128) {  // four windows of 32 in flight
          int32_t o[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int32_t q = q0 + 32 * j + lane;
            o[j] = q < xe ? g.ci[q] : -1;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (o[j] < 0) continue;
            if (pass == 0) {
              if (!h2_insert(htab, o[j] - base, size)) atomicOr(a.status, (int32_t)kSpillOverflow);
            } else {
              const uint32_t c = h2_count(htab, o[j] - base, size) - 1u;
              if (c && c < 1023u) {
                atomicAdd(&a.P[q0 + 32 * j + lane], (unsigned long long)c);  // slot (x, o)
                sx += c;
              }
            }
          }
        }
        if (pass == 1) {
          for (int off = 16; off; off >>= 1) sx += __shfl_xor_sync(0xffffffffu, sx, off);
          if (lane == 0 && sx) atomicAdd(&a.P[p], sx);  // slot (h, x)
        }
      }
      __syncthreads();
    }
  }
  if (lane == 0 && w_wedge) atomicAdd(&s_wedge, (unsigned long long)w_wedge);
  __syncthreads();
  if (threadIdx.x == 0 && s_wedge) {  // one atomic a block
    atomicAdd(a.work + kWorkCWedge, s_wedge);
    atomicAdd(a.work + kWorkCHash2Wedge, s_wedge);
  }
}

// ---------------- derive X_1..X_17 per graph ----------------
__device__ __forceinline__ bool div_exact(u128 num, u128 den, u128* q) {
  if (num % den != 0) return false;
  *q = num / den;
  return true;
}

__global__ void k_derive(int32_t G, const int32_t* __restrict__ gn, const int64_t* __restrict__ gm,
                         const unsigned long long* __restrict__ csum,
                         unsigned long long* __restrict__ xout, int32_t* __restrict__ status) {
  for (int32_t gi = blockIdx.x * blockDim.x + threadIdx.x; gi < G; gi += gridDim.x * blockDim.x) {
    u128 C[17];
    const int idx[13] = {3, 4, 5, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16};
    for (int k = 0; k < 13; ++k) {
      const unsigned long long* p = csum + ((size_t)gi * 13 + k) * 2;
      C[idx[k]] = ((u128)p[1] << 64) | (u128)p[0];
    }
    const u128 n = (u128)gn[gi], m = (u128)gm[gi];
    const u128 n2 = n < 2 ? 0 : n * (n - 1) / 2;
    const u128 n3 = n < 3 ? 0 : n2 * (n - 2) / 3;
    const u128 n4 = n < 4 ? 0 : n3 * (n - 3) / 4;
    u128 X[18];
    bool ok = true;
    X[1] = m;
    X[2] = n2 - m;
    ok &= div_exact(C[3], 3, &X[3]);
    ok &= div_exact(C[4], 2, &X[4]);
    X[5] = C[5];
    X[6] = n3 - X[3] - X[4] - X[5];
    ok &= div_exact(C[7], 6, &X[7]);
    X[8] = C[8] - C[7];
    ok &= div_exact(C[9] - 4 * X[8], 2, &X[9]);
    ok &= div_exact(C[10], 4, &X[10]);
    ok &= div_exact(C[11] - X[9], 3, &X[11]);
    X[12] = C[12] - C[10];
    ok &= div_exact(C[13] - X[9], 3, &X[13]);
    ok &= div_exact(C[14] - 6 * X[7] - 4 * X[8] - 2 * X[9] - 4 * X[10] - 2 * X[12], 2, &X[14]);
    ok &= div_exact(C[15] - 2 * X[12], 2, &X[15]);
    X[16] = C[16] - 2 * X[14];
    u128 s = 0;
    for (int i = 7; i <= 16; ++i) s += X[i];
    X[17] = n4 - s;
    for (int i = 1; i <= 17; ++i) {
      xout[((size_t)gi * 17 + (i - 1)) * 2] = (unsigned long long)X[i];
      xout[((size_t)gi * 17 + (i - 1)) * 2 + 1] = (unsigned long long)(X[i] >> 64);
    }
    if (!ok) atomicOr(status, (int32_t)kInexact);
  }
}

int g_grid = 0;

size_t smem_bytes(bool smem_table, int32_t table_n) {
  return smem_table ? sizeof(uint32_t) * (size_t)((table_n + 3) & ~3) : 0;
}

// The limit on a kernel's shared memory is the process's: every call sets it to the
// most the kernel ever takes, not to what its own graph needs, which another thread
// might be about to launch with more than.
template <typename K>
gc_status launch(K kernel, size_t smem, size_t most, const DevGraph& g, const CountArgs& a, cudaStream_t s,
                 const char* what) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return cuda_fail(e, what);
  int grid = count_grid_size();
  if (a.n_units < grid) grid = a.n_units > 0 ? a.n_units : 1;
  kernel<<<grid, kBlock, smem, s>>>(g, a);
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, what);
}

}  // namespace

// Persistent grid: kCtasPerSm CTAs of kBlock threads per SM.
int count_grid_size() {
  if (g_grid == 0) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    g_grid = (sms > 0 ? sms : 1) * kCtasPerSm;
  }
  return g_grid;
}

gc_status run_pass_c(const DevGraph& g, const CountArgs& a, cudaStream_t s) {
  const bool sm = a.tables == nullptr;
  if (sm) return launch(k_pass_c<true>, smem_bytes(true, g.table_n), smem_bytes(true, kSmemTableMax), g, a, s, "k_pass_c");
  return launch(k_pass_c<false>, 0, 0, g, a, s, "k_pass_c");
}

gc_status run_rows(const DevGraph& g, const CountArgs& a, cudaStream_t s) {
  if (g.n == 0) return GC_OK;
  k_rows<<<g.n, kRowBlock, smem_bytes(true, g.table_n), s>>>(g, a);  // at most 16 KB
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_rows");
}

gc_status run_rows_dense(const DevGraph& g, const CountArgs& a, cudaStream_t s) {
  k_rows_dense<<<g.n, kRowDenseBlock, 0, s>>>(g, a);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_rows_dense");
}

gc_status run_cliques_dense(const DevGraph& g, const CountArgs& a, int32_t kmax, cudaStream_t s) {
  const int32_t units = a.ktier_off[kNumTiers];
  if (units <= 0) return GC_OK;
  auto smem = [](int32_t k) { return 4 * ((size_t)k * dense_stride(k) + 2 * (size_t)k); };
  cudaError_t e = cudaFuncSetAttribute(k_cliques_dense, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem(kDenseMaxK));  // 140 KB, see launch()
  if (e != cudaSuccess) return cuda_fail(e, "k_cliques_dense");
  k_cliques_dense<<<units, kDenseBlock, smem(kmax), s>>>(g, a, kmax);
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_cliques_dense");
}

gc_status run_pass_c_heavy(const DevGraph& g, const CountArgs& a, cudaStream_t s) {
  if (a.n_cheavy <= 0 || !g.hgeom) return GC_OK;
  const size_t smem = sizeof(uint32_t) * (size_t)a.hub_tab;
  cudaError_t e = cudaFuncSetAttribute(k_pass_c_heavy, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return cuda_fail(e, "k_pass_c_heavy");
  int grid = count_grid_size() / kCtasPerSm;
  if (grid > a.n_cjobs) grid = a.n_cjobs;
  if (grid < 1) return GC_OK;
  k_pass_c_heavy<<<grid, kHeavyBlock, smem, s>>>(g, a);
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_pass_c_heavy");
}

template <int kThreads, int kMaxW>
static gc_status launch_hash(const DevGraph& g, const CountArgs& a, int32_t k0, int32_t k1, int32_t* cursor,
                             Fork* fork, int* launches) {
  if (k1 <= k0) return GC_OK;
  auto kern = k_pass_c_hash<kThreads, kMaxW>;
  const size_t smem = sizeof(int32_t) * 2 * kMaxW + sizeof(uint32_t) * kMaxW;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return cuda_fail(e, "k_pass_c_hash");
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem);
  if (e != cudaSuccess) return cuda_fail(e, "k_pass_c_hash occupancy");
  int grid = (per_sm > 0 ? per_sm : 1) * (count_grid_size() / kCtasPerSm);
  if (grid > k1 - k0) grid = k1 - k0;
  kern<<<grid, kThreads, smem, fork->next()>>>(g, a, k0, k1, cursor);
  ++*launches;
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_pass_c_hash");
}

gc_status run_pass_c_hash(const DevGraph& g, const CountArgs& a, Fork* fork, int* launches) {
  if (a.n_chash <= 0) return GC_OK;
  gc_status st = launch_hash<kHashBlock, kHashMaxW>(g, a, 0, a.n_chash_mid, a.cursor + 9, fork, launches);
  if (st != GC_OK) return st;
  st = launch_hash<kHashMidBlock, kHashMidW>(g, a, a.n_chash_mid, a.n_chash_big, a.cursor + 16, fork, launches);
  if (st != GC_OK) return st;
  return launch_hash<kHashSmallBlock, kHashSmallW>(g, a, a.n_chash_big, a.n_chash, a.cursor + 7, fork, launches);
}

template <int kThreads, int kSlots>
static gc_status launch_hash2(const DevGraph& g, const CountArgs& a, int32_t k0, int32_t k1, int32_t* cursor,
                              Fork* fork, int* launches) {
  if (k1 <= k0) return GC_OK;
  auto kern = k_pass_c_hash2<kThreads, kSlots>;
  const size_t smem = sizeof(uint32_t) * kSlots;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return cuda_fail(e, "k_pass_c_hash2");
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem);
  if (e != cudaSuccess) return cuda_fail(e, "k_pass_c_hash2 occupancy");
  int grid = (per_sm > 0 ? per_sm : 1) * (count_grid_size() / kCtasPerSm);
  if (grid > k1 - k0) grid = k1 - k0;
  kern<<<grid, kThreads, smem, fork->next()>>>(g, a, k0, k1, cursor);
  ++*launches;
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_pass_c_hash2");
}

gc_status run_pass_c_hash2(const DevGraph& g, const CountArgs& a, Fork* fork, int* launches) {
  if (a.n_chash2 <= 0) return GC_OK;
  gc_status st = launch_hash2<kHash2Block, kHash2Slots>(g, a, 0, a.n_chash2_big, a.cursor + 15, fork, launches);
  if (st != GC_OK) return st;
  return launch_hash2<kHash2Block / 2, kHash2HalfSlots>(g, a, a.n_chash2_big, a.n_chash2, a.cursor + 17, fork, launches);
}

gc_status run_finish(const DevGraph& g, const CountArgs& a, cudaStream_t s) {
  if (g.m == 0) return GC_OK;
  int blocks = (int)min((int64_t)count_grid_size() * 4, ((int64_t)g.m + kFinBlock - 1) / kFinBlock);
  if (a.per_edge_host) k_finish<true><<<blocks, kFinBlock, 0, s>>>(g, a);
  else k_finish<false><<<blocks, kFinBlock, 0, s>>>(g, a);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_finish");
}

gc_status run_induced(const DevGraph& g, const CountArgs& a, unsigned long long* vsum, uint64_t* out, bool out_host,
                      cudaStream_t s) {
  if (g.m == 0) return GC_OK;
  const int vblocks = (int)min((int64_t)count_grid_size() * 4, ((int64_t)g.n * 32 + 255) / 256);
  k_vertex_sums<<<vblocks > 0 ? vblocks : 1, 256, 0, s>>>(g, a.trio, vsum);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && g.n_long > 0) {
    k_vertex_sums_long<<<g.n_long, kLongRowBlock, 0, s>>>(g, a.trio, vsum);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return cuda_fail(e, "k_vertex_sums");
  const int blocks = (int)min((int64_t)count_grid_size() * 4, ((int64_t)g.m + kFinBlock - 1) / kFinBlock);
  unsigned long long* o = reinterpret_cast<unsigned long long*>(out);
  if (out_host) k_finish_induced<true><<<blocks, kFinBlock, 0, s>>>(g, a, vsum, o);
  else k_finish_induced<false><<<blocks, kFinBlock, 0, s>>>(g, a, vsum, o);
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_finish_induced");
}

gc_status run_derive(const DevGraph& g, const unsigned long long* csum, unsigned long long* x,
                     int32_t* status, cudaStream_t s) {
  int blocks = (g.G + 127) / 128;
  k_derive<<<blocks > 0 ? blocks : 1, 128, 0, s>>>(g.G, g.gn, g.gm, csum, x, status);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_derive");
}

}  // namespace gc
