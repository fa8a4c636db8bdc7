// gc_small.cu -- small graphs (n <= 1024) counted on a shared-memory
// adjacency bitmatrix.
//
// For a graph of at most 1024 vertices the whole adjacency fits in at most
// 132 KB of shared memory as bit rows. The paper's Psi marks with vertex
// types (Alg. 1: lambda1 for Gamma(v), lambda2 for S_u, lambda3 for T)
// become bit masks over the graph's vertices:
//   T = row(u) & row(v),  S_u = row(u) & ~row(v) without v,  S_v likewise,
// and |T| = popc(row(u) & row(v)), |S_u| = d_u - 1 - |T|, |S_v| and D_e
// follow per edge as in Sec. 4.5. The batched form returns only the global
// counts, so the per-edge summands of C_3 .. C_16 are needed only as sums
// over the edges: they are polynomials in |T|, d_u and d_v, and the kernel
// sums per edge only |T|, |T|^2, |T| (d_u + d_v) and d_u d_v, per vertex d^2
// and d^3, from which the columns follow in closed form (graph_column). Of the
// two per-edge scans of Alg. 5/6:
//   C_10 = sum_e x10 = 4 X_10 = 4 C4 - 4 C_8 + 2 C_7, with C4 the 4-cycles as
//          subgraphs, (1/2) sum over vertex pairs {u, w} of C(c_uw, 2) (c_uw
//          common neighbours; each cycle is met from both of its diagonals),
//          X_10 = C4 - X_8 - 3 X_7 and X_8 = C_8 - C_7 (Sec. 4.6). One pass over
//          the n^2 / 2 pairs, a lane per pair, gives c_uw and, where u ~ w,
//          |T| of the edge: no reduction over lanes per edge.
//   C_7  = sum_e x7  = 6 #K4: the 4-cliques with lowest vertex u are the
//          triangles of H_u, the subgraph induced on the k neighbours above u.
//          H_u is packed to k bits a row (a ballot per row and word) and its
//          triangles counted as sum over its edges (i, j), i < j, of the common
//          neighbours above j: k / 32 words a row instead of n / 32, and no
//          list of members per edge. A warp per u up to 128 neighbours above
//          it, the CTA together beyond. An H_u of few edges is counted edge by
//          edge instead (few_edges), one of fewer than three not at all.
// Rows are stored at an odd word stride, so that 32 lanes reading one word
// index of 32 rows hit 32 banks; four u's share the words of row w, five quarters
// of a read per 32 pairs and word. What bounds it: instruction issue, 86 % of the
// cycles in the classes above 128 vertices (shared-memory wavefronts 47 %, the
// pipe of popc 25 % of their peaks), with barriers in the smaller ones. (Before, each edge
// listed its common neighbours and took one of their rows at a time over the
// lanes: the graphs of n <= 512 in a launch of 48 took 5.3 ms, one CTA each;
// now 0.24 ms, in 256 parts.)
//
// Graphs are binned by vertex count into size classes (n <= 64, 128, 256,
// 512, 1024); each class runs its own instantiation, whose shared memory is
// sized for the class, so that small graphs take little and many CTAs fit on
// an SM. The block size of each class is a tuning parameter (BatchConfig). A
// CTA takes one unit at a time from the class's list, most work first: a
// graph, or, when a launch has too few graphs to fill the GPU, a part of one
// (every parts-th group of vertices u); each part loads the graph's bit rows, and the
// sums of a graph meet in global memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "gc_internal.h"

namespace gc {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// Sums of one graph from which its unrestricted sums follow in closed form
// (graph_column): per edge (u, v) with t = |T| and a = d_u + d_v, the sums of
// t, t^2, t a and d_u d_v; per vertex, d^2 and d^3; over vertex pairs,
// C(c_uw, 2); and the 4-cliques.
enum { kQt, kQtt, kQta, kQdd, kQd2, kQd3, kQc4, kQk4, kQn };
static_assert(kQn == kSmallSums, "sums of a small graph");

// The unrestricted sums of one graph (n vertices, m edges) from the sums q,
// in the column order
// C_3 C_4 C_5 C_7 C_8 C_9 C_10 C_11 C_12 C_13 C_14 C_15 C_16. Per edge
// |S_u| = d_u - 1 - t and |S_v| = d_v - 1 - t (Sec. 4.5), so s = a - 2 - 2t
// and D = n - 2 - t - s, and with A1 = sum a = sum_v d^2,
// A2 = sum a^2 = sum_v d^3 + 2P and P = sum over edges of d_u d_v:
//   C_4 = sum s = A1 - 2m - 2 sum t,       C_9 = sum t s = sum t a - 2 sum t - 2 sum t^2,
//   C_12 = sum |S_u||S_v| = P - A1 + m - sum t a + 2 sum t + sum t^2,
//   sum s^2 = A2 - 4 A1 + 4m - 4 (sum t a - 2 sum t) + 4 sum t^2,
//   C_5 = (n-2) m - sum t - C_4,            C_8 = (sum t^2 - sum t) / 2,
//   C_11 = (sum s^2 - 2 C_12 - C_4) / 2,    C_13 = (n-2) sum t - sum t^2 - C_9,
//   C_14 = m^2 + m - A1,                    C_15 = (n-2) C_4 - C_9 - sum s^2,
//   C_16 = (sum D^2 - C_5) / 2, sum D^2 = (n-2)^2 m - 2 (n-2)(sum t + C_4)
//          + sum t^2 + 2 C_9 + sum s^2,
// C_7 = 6 #K4, C_10 = 4 C4 - 4 C_8 + 2 C_7 with 2 C4 = sum over pairs of C(c_uw, 2).
// Column k of the graph, k in 0 .. 12. Unsigned arithmetic: every result is a nonnegative count below 2^64, so
// the wrap-around of the intermediate terms cancels.
__device__ __forceinline__ unsigned long long graph_column(int k, const unsigned long long* q, int32_t n, int64_t m) {
  typedef unsigned long long U;
  const U N2 = (U)(long long)(n - 2), M = (U)m;
  const U St = q[kQt], Stt = q[kQtt], Sta = q[kQta], A1 = q[kQd2];
  const U C4 = A1 - 2ull * M - 2ull * St;
  const U C9 = Sta - 2ull * St - 2ull * Stt;
  const U C12 = q[kQdd] - A1 + M - Sta + 2ull * St + Stt;
  const U Sss = q[kQd3] + 2ull * q[kQdd] - 4ull * A1 + 4ull * M - 4ull * (Sta - 2ull * St) + 4ull * Stt;
  const U C5 = N2 * M - St - C4;
  switch (k) {
    case 0: return St;
    case 1: return C4;
    case 2: return C5;
    case 3: return 6ull * q[kQk4];
    case 4: return (Stt - St) / 2ull;
    case 5: return C9;
    case 6: return 2ull * q[kQc4] - 2ull * (Stt - St) + 12ull * q[kQk4];
    case 7: return (Sss - 2ull * C12 - C4) / 2ull;
    case 8: return C12;
    case 9: return N2 * St - Stt - C9;
    case 10: return M * M + M - A1;
    case 11: return N2 * C4 - C9 - Sss;
    default: return (N2 * N2 * M - 2ull * N2 * (St + C4) + Stt + 2ull * C9 + Sss - C5) / 2ull;
  }
}

// Row stride of a size class: the words of a row, made odd.
__host__ __device__ constexpr int small_stride(int kN) { return (kN / 32) | 1; }

// H_u of up to 32 kWords members, packed: block b of 32 rows keeps the words
// b .. kWords - 1 of its rows (row i: the members j > i), at an odd stride.
__host__ __device__ constexpr int h_stride(int words, int b) { return (words - b) | 1; }
__host__ __device__ constexpr int h_words(int words) {
  int t = 0;
  for (int b = 0; b < words; ++b) t += 32 * h_stride(words, b);
  return t;
}
// Most members a warp takes alone.
__host__ __device__ constexpr int warp_members(int kN) { return kN < 128 ? kN : 128; }

// Shared memory of a size class, in bytes: the bitmatrix (kN rows at the odd
// stride), the H_u of every warp or the CTA's, the member lists of the same,
// the degrees, and the neighbours above each vertex.
__host__ __device__ constexpr size_t small_max(size_t a, size_t b) { return a > b ? a : b; }
__host__ __device__ constexpr size_t small_bm(int kN) { return (size_t)kN * (size_t)small_stride(kN) * 4; }
__host__ __device__ constexpr size_t small_h(int kN, int kBlock) {
  return 4 * small_max((size_t)(kBlock / 32) * h_words(warp_members(kN) / 32), h_words(kN / 32));
}
__host__ __device__ constexpr size_t small_list(int kN, int kBlock) {
  return 2 * small_max((size_t)(kBlock / 32) * warp_members(kN), (size_t)kN);
}
__host__ __device__ constexpr size_t small_smem(int kN, int kBlock) {
  return small_bm(kN) + small_h(kN, kBlock) + small_list(kN, kBlock) + 4 * (size_t)kN;
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long x) {
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Packs H_u (members m[0 .. k), ascending) into h from the bit rows bm, row
// stride kS; warp wi of nw takes every nw-th (row block, word).
template <int kS>
__device__ __forceinline__ void pack_h(const uint32_t* __restrict__ bm, const uint16_t* m, int k, uint32_t* h, int wi,
                                       int nw, int lane) {
  const int W = (k + 31) >> 5;
  int task = 0;
  for (int b = 0; b < W; ++b) {  // word b: members j = 32 b + lane
    const int j = 32 * b + lane;
    const int mj = j < k ? m[j] : 0;
    const int wj = mj >> 5, sj = 31 - (mj & 31);
    const uint32_t valid = k - 32 * b >= 32 ? kFull : (1u << (k - 32 * b)) - 1u;
    int off = 0;
    for (int rb = 0; rb <= b; ++rb, ++task) {  // rows i = 32 rb + r
      const int stride = h_stride(W, rb);
      if (task % nw == wi) {
        const int mi = 32 * rb + lane < k ? m[32 * rb + lane] : 0;
        const int rows = min(32, k - 32 * rb);
        uint32_t val = 0;
        for (int r = 0; r < rows; ++r) {
          const uint32_t word = bm[__shfl_sync(kFull, mi, r) * kS + wj];
          const uint32_t bits = __ballot_sync(kFull, (int32_t)(word << sj) < 0);
          if (lane == r) val = bits;
        }
        val &= valid;
        if (rb == b) val &= lane == 31 ? 0u : kFull << (lane + 1);  // members above the row's
        h[off + lane * stride + (b - rb)] = val;
      }
      off += 32 * stride;
    }
  }
}

// This lane's part of the triangles of the packed H_u: for every pair (i, j),
// j = 32 b + lane, with bit j of row i set, the common members above j.
__device__ __forceinline__ uint32_t count_h(const uint32_t* h, int k, int wi, int nw, int lane) {
  const int W = (k + 31) >> 5;
  uint32_t acc = 0;
  int task = 0, offb = 0;
  for (int b = 0; b < W; ++b) {
    const uint32_t* hj = h + offb + lane * h_stride(W, b);  // words b .. W - 1 of row j
    int off = 0;
    for (int rb = 0; rb <= b; ++rb, ++task) {
      const int stride = h_stride(W, rb);
      if (task % nw == wi) {
        const uint32_t* hi0 = h + off + (b - rb);  // word b of row 32 rb
        const int rows = min(32, k - 32 * rb);
        for (int w = b; w < W; w += 4) {
          uint32_t x[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = w + q < W ? hj[w - b + q] : 0u;
          const uint32_t* hi = hi0;
          for (int r = 0; r < rows; ++r, hi += stride) {
            const uint32_t on = 0u - ((hi[0] >> lane) & 1u);  // all ones when i ~ j
            uint32_t c = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (w + q < W) c += __popc(hi[w - b + q] & x[q]);  // warp-uniform
            acc += c & on;
          }
        }
      }
      off += 32 * stride;
    }
    offb += 32 * h_stride(W, b);
  }
  return acc;
}

// This lane's part of the 4-cliques with lowest vertex u, edge by edge of H_u:
// a lane per member v, its edges (v, w) one after the other, the common
// neighbours above w of each. For an H_u of few edges: the neighbourhoods of a
// star's centre or of one side of a bipartite graph have none, and packing a
// k x k matrix for each of them was most of such a graph's time.
template <int kS>
__device__ __noinline__ uint32_t count_edges(const uint32_t* __restrict__ bm, const uint32_t* __restrict__ ru,
                                                const int32_t* __restrict__ above, int k, int W, int lane) {
  uint32_t acc = 0;
  for (int i = lane; i < k; i += 32) {
    const int v = above[i];
    const uint32_t* rv = bm + v * kS;
    uint32_t keep = (kFull << (v & 31)) << 1;  // ids above v
    for (int a = v >> 5; a < W; ++a, keep = kFull) {
      uint32_t t = ru[a] & rv[a] & keep;
      while (t) {
        const int b = __ffs(t) - 1;
        t &= t - 1u;
        const uint32_t* rw = bm + (32 * a + b) * kS;
        uint32_t hi = (kFull << b) << 1;
        for (int c = a; c < W; ++c, hi = kFull) acc += __popc(ru[c] & rv[c] & rw[c] & hi);
      }
    }
  }
  return acc;
}
// Whether H_u, k members and at most e edges, is counted edge by edge rather
// than packed, by SM cycles: about W / 4 a member and 2 W an edge against k / 24
// a member and k^2 / 1500 a pair (small_cost).
__device__ __forceinline__ bool few_edges(int k, uint32_t e, int W) {
  const float K = (float)k;
  return (float)W * (0.25f * K + 2.0f * (float)e) < K * K * (1.0f / 24.0f + K * (1.0f / 1500.0f));
}
constexpr uint16_t kFewEdges = 0x8000;  // in s_up

// The pairs of kU consecutive vertices u0, u0 + 1, ... with the vertices above
// them, a lane per w: every word of row w is loaded once for all of them. (One u
// at a time: 2000 graphs of 1000 vertices and mean degree 5 took 14.9 ms, now 9.5.) Lane i
// adds sum i of them to `mine`: sums over four u stay in 32 bits (4092 pairs at
// most, c and the degrees at most 1023). Marks the u that need no H_u, and those
// whose H_u is counted edge by edge.
template <int kS, int kU>
__device__ __forceinline__ void small_pairs(const uint32_t* __restrict__ bm, const uint16_t* __restrict__ deg,
                                            uint16_t* __restrict__ up, int u0, int n, int W, int lane,
                                            unsigned long long& mine) {
  const uint32_t* rowu = bm + u0 * kS;
  uint32_t at[kU], tt = 0, tw = 0, dd = 0, c4 = 0;
#pragma unroll
  for (int i = 0; i < kU; ++i) at[i] = 0u;
  for (int w0 = u0 + 1; w0 < n; w0 += 32) {
    const int w = w0 + lane;
    if (w >= n) continue;
    const uint32_t* roww = bm + w * kS;
    uint32_t c[kU];
#pragma unroll
    for (int i = 0; i < kU; ++i) c[i] = 0u;
#pragma unroll 2
    for (int k = 0; k < W; ++k) {
      const uint32_t x = roww[k];
#pragma unroll
      for (int i = 0; i < kU; ++i) c[i] += __popc(rowu[i * kS + k] & x);  // rows past n: of the array, not used
    }
    const uint32_t dw = deg[w];
    const int ww = w >> 5, wb = w & 31;
#pragma unroll
    for (int i = 0; i < kU; ++i) {
      if (w <= u0 + i) continue;  // also u0 + i >= n
      c4 += c[i] * (c[i] - 1u) / 2u;  // 0 for c = 0: the product is 0
      if ((rowu[i * kS + ww] >> wb) & 1u) {
        at[i] += c[i];
        tt += c[i] * c[i];
        tw += c[i] * dw;
        dd += deg[u0 + i] * dw;
      }
    }
  }
  unsigned long long t = 0, ta = 0;
#pragma unroll
  for (int i = 0; i < kU; ++i) {
    const uint32_t ti = __reduce_add_sync(kFull, at[i]);  // at least twice the edges of H_u
    t += ti;
    if (u0 + i < n) {  // warp-uniform
      ta += (unsigned long long)deg[u0 + i] * ti;
      if (lane == 0) {
        if (ti < 6u) up[u0 + i] = 0;  // fewer than three edges: no triangle in H_u
        else if (few_edges(up[u0 + i], ti / 2u, W)) up[u0 + i] |= kFewEdges;
      }
    }
  }
  const uint32_t d = lane < kU && u0 + lane < n ? deg[u0 + lane] : 0u;
  if (lane == kQt) mine += t;
  auto add = [&](int i, uint32_t v, unsigned long long more = 0ull) {
    v = __reduce_add_sync(kFull, v);
    if (lane == i) mine += v + more;
  };
  add(kQtt, tt);
  add(kQta, tw, ta);
  add(kQdd, dd);
  add(kQd2, d * d);
  add(kQd3, d * d * d);
  add(kQc4, c4);
}

// at least 1536 threads resident per SM (at most 42 registers a thread) where
// shared memory has room for them: the more warps an SM holds, the more of its
// cycles issue
__host__ __device__ constexpr int small_ctas(int kN, int kBlock) {
  const int fit = (int)(((size_t)227 << 10) / (small_smem(kN, kBlock) + 3072));
  return fit < 1 ? 1 : fit < 1536 / kBlock ? fit : 1536 / kBlock;
}
template <int kN, int kBlock>
__global__ void __launch_bounds__(kBlock, small_ctas(kN, kBlock)) k_small_graphs(const int32_t* __restrict__ rp,
                                                         const int64_t* __restrict__ voff,
                                                         const int32_t* __restrict__ ci,
                                                         const int64_t* __restrict__ eoff,
                                                         const int2* __restrict__ units, int32_t n_units,
                                                         int32_t* __restrict__ cursor, int32_t* __restrict__ status,
                                                         unsigned long long* __restrict__ sums) {
  constexpr int kS = small_stride(kN);  // words per bit row, odd
  constexpr int kWarps = kBlock / 32;
  constexpr int kWarpK = warp_members(kN);
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* bm = reinterpret_cast<uint32_t*>(smem);
  uint32_t* s_h = reinterpret_cast<uint32_t*>(smem + small_bm(kN));
  uint16_t* s_m = reinterpret_cast<uint16_t*>(smem + small_bm(kN) + small_h(kN, kBlock));
  uint16_t* s_deg = reinterpret_cast<uint16_t*>(smem + small_bm(kN) + small_h(kN, kBlock) + small_list(kN, kBlock));
  uint16_t* s_up = s_deg + kN;
  __shared__ int32_t s_unit;
  __shared__ unsigned long long s_q[kBlock / 32][kQn];  // per warp: a 64-bit shared atomic is a loop of compare-and-swaps
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_unit = atomicAdd(cursor, 1);
    __syncthreads();
    if (s_unit >= n_units) break;
    const int2 unit = units[s_unit];  // graph, part | parts << 16
    const int32_t g = unit.x, part = unit.y & 0xffff, parts = unit.y >> 16;
    const int32_t* grp = rp + voff[g];
    const int32_t* gci = ci + eoff[g];
    const int32_t n = (int32_t)(voff[g + 1] - voff[g]) - 1;
    if (n > kN) {  // cannot happen: graphs are binned by n
      if (threadIdx.x == 0) atomicOr(status, (int32_t)kSpillOverflow);
      continue;
    }
    const int W = (n + 31) / 32;
    for (int32_t i = threadIdx.x; i < n * kS; i += kBlock) bm[i] = 0u;
    __syncthreads();
    // the bit rows, the degrees, and the neighbours above each vertex
    // (four rows of a warp at a time, their first 32 entries in flight together:
    // one row after the other, this was half of a sparse graph's time)
    constexpr int kRows = 4;
    for (int32_t x0 = kRows * warp; x0 < n; x0 += kRows * kWarps) {
      const int32_t off = lane <= kRows ? grp[min(x0 + lane, n)] : 0;
      int32_t xb[kRows], len[kRows], y[kRows], up[kRows];
#pragma unroll
      for (int j = 0; j < kRows; ++j) {  // rows past n are empty
        xb[j] = __shfl_sync(kFull, off, j);
        len[j] = __shfl_sync(kFull, off, j + 1) - xb[j];
        y[j] = lane < len[j] ? gci[xb[j] + lane] : -1;
      }
#pragma unroll
      for (int j = 0; j < kRows; ++j) {
        const int32_t x = x0 + j;
        if (y[j] >= 0) atomicOr(&bm[x * kS + (y[j] >> 5)], 1u << (y[j] & 31));
        up[j] = __popc(__ballot_sync(kFull, y[j] > x));
        for (int32_t k = 32; k < len[j]; k += 32) {
          const int32_t z = k + lane < len[j] ? gci[xb[j] + k + lane] : -1;
          if (z >= 0) atomicOr(&bm[x * kS + (z >> 5)], 1u << (z & 31));
          up[j] += __popc(__ballot_sync(kFull, z > x));
        }
        if (lane == 0 && x < n) {
          s_deg[x] = (uint16_t)len[j];
          s_up[x] = (uint16_t)up[j];
        }
      }
    }
    __syncthreads();
    // this unit's vertices u, groups of kU in turn: part, part + parts, ..., one
    // per warp: four where every warp gets several, else one
    const int32_t turn = parts * kWarps, first = part + parts * warp;
    const int32_t group = n >= 4 * turn ? 4 : 1;
    unsigned long long mine = 0;  // lane i: sum i
    for (int32_t u = group * first; u < n; u += group * turn) {
      if (group == 4) small_pairs<kS, 4>(bm, s_deg, s_up, u, n, W, lane, mine);
      else small_pairs<kS, 1>(bm, s_deg, s_up, u, n, W, lane, mine);
    }
    if (lane < kQk4) s_q[warp][lane] = mine;
    __syncthreads();  // the marks in s_up
    // the 4-cliques with lowest vertex u: the triangles of H_u
    unsigned long long q_k4 = 0;
    {
      uint32_t* h = s_h + warp * h_words(kWarpK / 32);
      uint16_t* m = s_m + warp * kWarpK;
      for (int32_t j = warp;; j += kWarps) {  // this unit's vertices one to a warp: the first have the most members
        const int32_t u = group * (part + parts * (j / group)) + j % group;
        if (u - j % group >= n) break;
        const int up = u < n ? s_up[u] : 0, k = up & ~kFewEdges;
        if (k < 3) continue;  // warp-uniform
        const int32_t p1 = grp[u + 1] - k;  // the neighbours above u end its ascending row
        if (up & kFewEdges) {
          q_k4 += count_edges<kS>(bm, bm + u * kS, gci + p1, k, W, lane);
          continue;
        }
        if (k > kWarpK) continue;
        for (int i = lane; i < k; i += 32) m[i] = (uint16_t)gci[p1 + i];
        __syncwarp();
        pack_h<kS>(bm, m, k, h, 0, 1, lane);
        __syncwarp();
        q_k4 += count_h(h, k, 0, 1, lane);
        __syncwarp();
      }
    }
    if (kN > kWarpK) {
      for (int32_t u0 = group * part; u0 < n; u0 += group * parts)
        for (int32_t u = u0; u < min(u0 + group, n); ++u) {
          const int k = s_up[u];
          if (k <= kWarpK || (k & kFewEdges)) continue;  // CTA-uniform
          __syncthreads();
          const int32_t p1 = grp[u + 1] - k;
          for (int i = threadIdx.x; i < k; i += kBlock) s_m[i] = (uint16_t)gci[p1 + i];
          __syncthreads();
          pack_h<kS>(bm, s_m, k, s_h, warp, kWarps, lane);
          __syncthreads();
          q_k4 += count_h(s_h, k, warp, kWarps, lane);
        }
    }
    q_k4 = warp_sum(q_k4);
    if (lane == 0) s_q[warp][kQk4] = q_k4;
    __syncthreads();
    if (threadIdx.x < kQn) {
      unsigned long long v = 0;
      for (int w = 0; w < kWarps; ++w) v += s_q[w][threadIdx.x];
      if (v) atomicAdd(&sums[(size_t)g * kQn + threadIdx.x], v);
    }
  }
}

// The unrestricted sums of every graph: thread per (graph, column).
__global__ void k_small_columns(int32_t G, const int32_t* __restrict__ gn, const int64_t* __restrict__ gm,
                                const unsigned long long* __restrict__ sums, unsigned long long* __restrict__ csum) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)G * 13) return;
  const int32_t g = (int32_t)(t / 13), k = (int32_t)(t % 13);
  csum[2 * t] = graph_column(k, sums + (size_t)g * kQn, gn[g], gm[g]);
  csum[2 * t + 1] = 0ull;
}

typedef void (*SmallKernel)(const int32_t*, const int64_t*, const int32_t*, const int64_t*, const int2*, int32_t,
                            int32_t*, int32_t*, unsigned long long*);

// kSmallBlocks[j] threads per CTA for tuning choice j.
constexpr int kNumSmallBlocks = 4;
constexpr int kSmallBlocks[kNumSmallBlocks] = {64, 128, 256, 512};

template <int kN>
SmallKernel small_kernel_for(int block) {
  switch (block) {
    case 64: return k_small_graphs<kN, 64>;
    case 128: return k_small_graphs<kN, 128>;
    case 512: return k_small_graphs<kN, 512>;
    default: return k_small_graphs<kN, 256>;
  }
}

SmallKernel small_kernel(int cls, int block) {
  switch (cls) {
    case 0: return small_kernel_for<64>(block);
    case 1: return small_kernel_for<128>(block);
    case 2: return small_kernel_for<256>(block);
    case 3: return small_kernel_for<512>(block);
    default: return small_kernel_for<1024>(block);
  }
}

int valid_block(int block) {
  for (int b : kSmallBlocks)
    if (b == block) return block;
  return 256;
}

}  // namespace

int small_class_of(int32_t n) {
  for (int c = 0; c < kSmallClasses; ++c)
    if (n <= kSmallClassN[c]) return c;
  return kSmallClasses;
}

// Resident CTAs of every (size class, block) instantiation on one GPU
// (filled by small_graphs_setup, outside any stream capture).
static int g_small_ctas[kSmallClasses][kNumSmallBlocks] = {};

static int block_index(int block) {
  for (int j = 0; j < kNumSmallBlocks; ++j)
    if (kSmallBlocks[j] == block) return j;
  return 2;
}

// Grid of one size class: resident CTAs, at most one CTA per unit.
static int small_grid(int cls, int block, int32_t units) {
  int grid = g_small_ctas[cls][block_index(block)];
  if (grid < 1) grid = 1;
  return grid > units ? units : grid;
}

// Cost of a graph in SM cycles, roughly (n = 500 at density 0.275 measures
// about 4e5): two cycles per 32 vertex pairs and word; H_u for k neighbours
// above u, k spread evenly over [0, 2 m / n], at k^2 / 64 ballots and k^3 /
// 6144 words of 32 pairs; and the bit rows.
static double small_cost(int32_t n, int64_t m) {
  const double W = (n + 31) / 32, k = n > 0 ? (double)m / n : 0.0;
  return (double)n * n * W / 32 + n * (k * k / 18 + k * k * k / 750 + 20) + (double)m / 4;
}

void small_units(const std::vector<int32_t>& n, const std::vector<int64_t>& m, std::vector<int2>* units,
                 int32_t* class_off) {
  const int32_t G = (int32_t)n.size();
  std::vector<double> cost((size_t)G);
  double total = 0;
  for (int32_t g = 0; g < G; ++g) total += cost[(size_t)g] = small_cost(n[(size_t)g], m[(size_t)g]);
  // A graph is cut into parts when it would be a long single tail, or when
  // the launch has too few graphs for the GPU: parts of about an eighth of an
  // SM's share, but no smaller than kLeast, since each part loads all bit rows
  // again. 48 graphs of n in [20, 500]: 5.9 ms uncut.
  constexpr double kLeast = 25000;
  const double target = std::max(kLeast, total / (8.0 * (count_grid_size() / kCtasPerSm)));
  // lists by class and by cost, eight bins to a factor of two, largest first
  constexpr int kBins = 512;
  std::vector<int32_t> at((size_t)kSmallClasses * kBins + 1, 0);
  std::vector<int32_t> bin((size_t)G), parts((size_t)G);
  for (int32_t g = 0; g < G; ++g) {
    const double c = cost[(size_t)g];
    const int k = c > 2 * target ? (int)std::min(32.0, c / target) : 1;
    const int lg = (int)(8 * std::log2(std::max(1.0, c / k)));
    parts[(size_t)g] = k;
    bin[(size_t)g] = small_class_of(n[(size_t)g]) * kBins + kBins - 1 - std::min(lg, kBins - 1);
    at[(size_t)bin[(size_t)g] + 1] += k;
  }
  for (size_t i = 1; i < at.size(); ++i) at[i] += at[i - 1];
  for (int c = 0; c <= kSmallClasses; ++c) class_off[c] = at[(size_t)c * kBins];
  units->resize((size_t)at.back());
  for (int32_t g = 0; g < G; ++g)
    for (int p = 0; p < parts[(size_t)g]; ++p)
      (*units)[(size_t)at[(size_t)bin[(size_t)g]]++] = make_int2(g, p | (parts[(size_t)g] << 16));
}

gc_status small_graphs_setup() {
  static std::mutex mu;
  static std::vector<int> done;  // devices
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lk(mu);
  if (e == cudaSuccess && std::find(done.begin(), done.end(), dev) != done.end()) return GC_OK;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_fail(e, "k_small_graphs setup");
  for (int c = 0; c < kSmallClasses; ++c)
    for (int j = 0; j < kNumSmallBlocks; ++j) {
      const int b = kSmallBlocks[j];
      const size_t smem = small_smem(kSmallClassN[c], b);
      e = cudaFuncSetAttribute(small_kernel(c, b), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      int per_sm = 0;
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, small_kernel(c, b), b, smem);
      if (e != cudaSuccess) return cuda_fail(e, "k_small_graphs attribute");
      g_small_ctas[c][j] = (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
    }
  done.push_back(dev);
  return GC_OK;
}

gc_status run_small_graphs(const SmallGraphs& b, const int32_t* class_off, const BatchConfig& cfg, cudaEvent_t* ev,
                           const SmallFork* fork, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  if (fork && (e = cudaEventRecord(fork->start, s)) != cudaSuccess) return cuda_fail(e, "small fork");
  for (int c = kSmallClasses - 1; c >= 0; --c) {  // the largest graphs first
    const int32_t units = class_off[c + 1] - class_off[c];
    if (ev && (e = cudaEventRecord(ev[2 * c], s)) != cudaSuccess) return cuda_fail(e, "small event");
    if (units > 0) {
      cudaStream_t sc = s;
      if (fork) {
        sc = fork->stream[c];
        if ((e = cudaStreamWaitEvent(sc, fork->start, 0)) != cudaSuccess) return cuda_fail(e, "small fork");
      }
      const int block = valid_block(cfg.class_block[c]);
      const int grid = small_grid(c, block, units);
      small_kernel(c, block)<<<grid, block, small_smem(kSmallClassN[c], block), sc>>>(
          b.rp, b.voff, b.ci, b.eoff, b.units + class_off[c], units, b.cursor + c, b.status, b.sums);
      if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "k_small_graphs");
      if (fork) {
        if ((e = cudaEventRecord(fork->done[c], sc)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(s, fork->done[c], 0)) != cudaSuccess)
          return cuda_fail(e, "small join");
      }
    }
    if (ev && (e = cudaEventRecord(ev[2 * c + 1], s)) != cudaSuccess) return cuda_fail(e, "small event");
  }
  const int64_t cols = (int64_t)b.G * 13;
  if (cols > 0) k_small_columns<<<(int)((cols + 255) / 256), 256, 0, s>>>(b.G, b.gn, b.gm, b.sums, b.csum);
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_small_columns");
}

}  // namespace gc
