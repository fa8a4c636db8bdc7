// gc_prep.cu -- one-time device preparation of an uploaded graph.
//
//   * degrees d_x and the P3 orientation of every edge (Sec. 4.3): the "low"
//     endpoint u has the smaller (degree, id) pair, the "high" endpoint v the
//     larger, so d_v >= d_u;
//   * the slot -> edge id map of both CSR directions (edge id: rank of (u, v),
//     u < v, in row-major upper-triangle order of the caller's labels);
//   * degree-oriented out-lists: out(x) = neighbours of higher (degree, id)
//     rank, ascending ids, the end of row x since ids are ranks. Each pair {a, b} of adjacent vertices appears in
//     exactly one out-list; the 4-clique step uses this to count each pair
//     of T once (the role of the Psi reset in Alg. 5);
//   * the work units of the counting passes: every vertex v that is the high
//     endpoint of at least one edge forms one "v-group" (its low neighbours);
//     groups are binned by floor(log2(estimated work)) and listed heaviest
//     bin first -- the difficulty-ordered edge queue Pi of Sec. 4.4 at group
//     granularity -- and split into the kernels of pass C by their wedges.
#include <cuda_runtime.h>

#include <cmath>

#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <vector>

#include "gc_internal.h"

namespace gc {
namespace {

constexpr int kScanTile = 2048;  // elements per scan tile (256 threads x 8)

// first index in [lo, hi) with a[i] >= key
__device__ __forceinline__ int32_t lower_bound_i32(const int32_t* a, int32_t lo, int32_t hi,
                                                   int32_t key) {
  while (lo < hi) {
    int32_t mid = lo + ((hi - lo) >> 1);
    if (a[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Degrees, out-degrees k (ids are ranks, so the higher-rank neighbours of x are
// the entries above x), the largest of both, and the sums of d^2 and of k (d - k).
__global__ void __launch_bounds__(256) k_deg_out(int32_t n, const int32_t* __restrict__ rp,
                                                 const int32_t* __restrict__ ci, int32_t* __restrict__ deg,
                                                 int32_t* __restrict__ out_cnt, int32_t* __restrict__ dmax,
                                                 int32_t* __restrict__ kmax, unsigned long long* __restrict__ sums) {
  int32_t dm = 0, km = 0;
  unsigned long long d2 = 0, kd = 0;
  for (int32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x) {
    const int32_t b = rp[x], e = rp[x + 1];
    const int32_t k = e - lower_bound_i32(ci, b, e, x + 1);
    deg[x] = e - b;
    out_cnt[x] = k;
    dm = max(dm, e - b);
    km = max(km, k);
    d2 += (unsigned long long)(e - b) * (unsigned)(e - b);
    kd += (unsigned long long)k * (unsigned)(e - b - k);
  }
  // one atomic a block and maximum: one a vertex on the same word took 0.8 ms
  // of the preparation of R-MAT scale 20
  __shared__ int32_t s_m[2];
  __shared__ unsigned long long s_s[2];
  if (threadIdx.x < 2) {
    s_m[threadIdx.x] = 0;
    s_s[threadIdx.x] = 0ull;
  }
  __syncthreads();
  dm = __reduce_max_sync(0xffffffffu, dm);
  km = __reduce_max_sync(0xffffffffu, km);
  for (int o = 16; o; o >>= 1) {
    d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    kd += __shfl_xor_sync(0xffffffffu, kd, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&s_m[0], dm);
    atomicMax(&s_m[1], km);
    atomicAdd(&s_s[0], d2);
    atomicAdd(&s_s[1], kd);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_m[0]) atomicMax(dmax, s_m[0]);
    if (s_m[1]) atomicMax(kmax, s_m[1]);
    if (s_s[0]) atomicAdd(&sums[0], s_s[0]);
    if (s_s[1]) atomicAdd(&sums[1], s_s[1]);
  }
}

// Warp per vertex x: the out-list, and the reverse slot of both directions of
// each of its edges, by one search in the higher end's row. eid (optional):
// the relabel wrote the id of the slot whose caller labels (perm) ascend; the
// other slot of the edge takes it here, and e2o the edge's out-slot.
__global__ void k_edges(int32_t n, int32_t m, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                        const int32_t* __restrict__ out_ptr, int32_t* __restrict__ eid,
                        int32_t* __restrict__ out_idx, int32_t* __restrict__ ocsr, int32_t* __restrict__ rev,
                        int32_t* __restrict__ e2o, const int32_t* __restrict__ perm) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t xw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; xw < n; xw += warps) {
    const int32_t x = (int32_t)xw;
    const int32_t e = rp[x + 1], o0 = out_ptr[x], k = out_ptr[x + 1] - o0;
    for (int32_t i = lane; i < k; i += 32) {
      const int32_t p = e - k + i, os = o0 + i;  // the entries above x end its row
      const int32_t y = ci[p];
      out_idx[os] = y;
      ocsr[os] = p;
      const int32_t yb = rp[y], ye = rp[y + 1];
      const int32_t q = lower_bound_i32(ci, yb, ye, x);
      const bool found = q < ye && ci[q] == x;
      if (found) {
        rev[p] = q;
        rev[q] = p;
      }  // else both keep rev = self (k_rev_init): no reverse, invalid input
      if (!eid) continue;
      int32_t ide;
      if (found && perm[x] > perm[y]) {
        ide = eid[q];
        eid[p] = ide;
      } else {
        ide = eid[p];
        if (found) eid[q] = ide;
      }
      if ((uint32_t)ide < (uint32_t)m) e2o[ide] = os;  // out of range only for invalid input
    }
  }
}

// rev[p] = p for every slot, before k_edges searches each edge once: a slot
// that no search reaches keeps it (it has no reverse).
__global__ void k_rev_init(int64_t nnz, int32_t* __restrict__ rev) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x)
    rev[p] = (int32_t)p;
}

// Edge list in the caller's labels when the graph was relabelled.
__global__ void k_uv_perm(int32_t n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                          const int32_t* __restrict__ eid, const int32_t* __restrict__ perm,
                          int32_t* __restrict__ uv) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int32_t x = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < n; x += warps) {
    const int32_t px = perm[x];
    for (int32_t p = rp[x] + lane; p < rp[x + 1]; p += 32) {
      const int32_t y = ci[p];
      if (y < x) continue;
      const int32_t py = perm[y];
      const int64_t e = eid[p];
      uv[2 * e] = px < py ? px : py;
      uv[2 * e + 1] = px < py ? py : px;
    }
  }
}

__device__ __forceinline__ int bin_of(long long cost) {
  return cost <= 1 ? 0 : 63 - __clzll(cost);
}

// Bin key of a v-group under the chosen ordering (0 volume, 1 degree, 2 none).
// Only the order of the units on the vertex-indexed tables depends on it (hub
// and hashed units are sorted by their wedges): the volume is taken as d^2.
__device__ __forceinline__ int unit_bin(int key, int32_t d) {
  return key == 0 ? bin_of((long long)d * d) : (key == 1 ? bin_of(d) : 0);
}

// Counts, or (kScatter) puts at places by bin from cursor[], the items 0 .. n - 1
// (bin < 0: left out): one atomic a block and bin.
template <int kBins, bool kScatter, class Bin, class Put>
__device__ __forceinline__ void bin_vertices(int32_t n, int32_t* __restrict__ cursor, Bin bin, Put put) {
  __shared__ int32_t h[kBins], base[kBins];
  for (int32_t v0 = blockIdx.x * blockDim.x; v0 < n; v0 += gridDim.x * blockDim.x) {
    for (int i = threadIdx.x; i < kBins; i += blockDim.x) h[i] = 0;
    __syncthreads();
    const int32_t v = v0 + threadIdx.x;
    const int b = v < n ? bin(v) : -1;
    int at = 0;
    if (b >= 0) at = atomicAdd(&h[b], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < kBins; i += blockDim.x)
      if (h[i]) base[i] = atomicAdd(&cursor[i], h[i]);
    __syncthreads();
    if (kScatter && b >= 0) put(base[b] + at, v);
    __syncthreads();
  }
}
template <bool kScatter>
__global__ void __launch_bounds__(1024) k_bin_units(int32_t n, const int32_t* __restrict__ deg,
                                                    const int32_t* __restrict__ out_cnt, int32_t* __restrict__ cursor,
                                                    int32_t* __restrict__ units, int key) {
  bin_vertices<64, kScatter>(
      n, cursor, [&](int32_t v) { return deg[v] - out_cnt[v] > 0 ? unit_bin(key, deg[v]) : -1; },
      [&](int32_t at, int32_t v) { units[at] = v; });
}

// Pass K units: every vertex a with |out(a)| = k >= 2 (a triangle needs two
// higher-rank neighbours), binned by ceil(log2 k) and listed largest bin
// first, so that the tiers of pass K (k > 1024, <= 1024, <= 512, <= 256,
// <= 32) are contiguous ranges of the list.
__device__ __forceinline__ int kbin_of(int32_t k) { return 32 - __clz(k - 1); }

template <bool kScatter>
__global__ void __launch_bounds__(1024) k_bin_kunits(int32_t n, const int32_t* __restrict__ out_cnt,
                                                     int32_t* __restrict__ cursor, int32_t* __restrict__ units) {
  bin_vertices<32, kScatter>(
      n, cursor, [&](int32_t v) { return out_cnt[v] >= 2 ? kbin_of(out_cnt[v]) : -1; },
      [&](int32_t at, int32_t v) { units[at] = v; });
}

// Pass-C units by kernel and wedges W: eight bins to a factor of two of W - 1
// (so that 512, 2048 and 8192 wedges end bins), for the hash, the two instances
// of the packed-key hash, and one bin for the vertex-indexed tables.
constexpr int kHashBins = 88, kHash2Bins = 24;
constexpr int kBinHalf = kHashBins, kBinBig = kBinHalf + kHash2Bins, kBinRest = kBinBig + kHash2Bins;
constexpr int kCBins = kBinRest + 1;
__host__ __device__ __forceinline__ int wedge_bin(int32_t w) {  // 1 <= w <= kHash2MaxW
  const int32_t v = w - 1;
  if (v < 8) return v;
  int o = 3;
  while ((v >> (o + 1)) != 0) ++o;
  return 8 * (o - 2) + ((v >> (o - 3)) & 7);
}
struct HubUnit {
  int32_t h, nx;
  long long w;
};

// Warp per unit h: its lower neighbours nx and wedges W = sum over them, x, of
// |{o in Gamma(x) : o < h}|. Ids are ranks and rows ascend, so the o < h of
// Gamma(x) are the entries before the slot of (x, h), the reverse of the slot of
// (h, x): no search per lower neighbour (the reverse is clamped into the row, as
// the hub kernel does, so that W is what the kernels count even before symmetry
// is checked). Then the unit's kernel: a hub unit pays, per shared-memory block
// of the o-range, a few microseconds of barriers (more when it has more than a
// CTA's worth of lower neighbours), against roughly 10 ns per wedge on an SM
// for a wedge on a vertex-indexed table in DRAM, so the hub kernel is taken
// when the wedges exceed blocks x max(1024, nx), tested from 16384 wedges, after
// both hashes have taken what fits them. Hub units are listed for the host, the
// others get their bin; units without wedges add nothing to P and are left out
// (bin -1). (The host used to make these lists from W and nx of every unit: 3 ms
// of an upload of R-MAT scale 20.)
__global__ void __launch_bounds__(256) k_cwork(int32_t n_units, const int32_t* __restrict__ units,
                                               const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                               const int32_t* __restrict__ rev, const int32_t* __restrict__ vgid,
                                               const int32_t* __restrict__ gbase, int32_t tab, bool packed,
                                               int32_t* __restrict__ bin, int32_t* __restrict__ hw,
                                               int32_t* __restrict__ hist, HubUnit* __restrict__ hubs) {
  __shared__ int32_t s_hist[kCBins];
  for (int i = threadIdx.x; i < kCBins; i += 256) s_hist[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * 256) >> 5;
  for (int32_t k = (int32_t)((blockIdx.x * 256 + threadIdx.x) >> 5); k < n_units; k += warps) {
    const int32_t h = units[k];
    const int32_t hb = rp[h];
    const int32_t nx = lower_bound_i32(ci, hb, rp[h + 1], h) - hb;
    long long w = 0;
    for (int32_t i = lane; i < nx; i += 32) {
      const int32_t x = ci[hb + i];
      const int32_t xb = rp[x];
      w += min(max(rev[hb + i], xb), rp[x + 1]) - xb;
    }
    for (int o = 16; o; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if (lane != 0) continue;
    int b = -1;
    if (w > 0 && w <= kHashMaxW) {
      b = wedge_bin((int32_t)w);
    } else if (w > 0 && w <= kHash2MaxW && nx < kHash2MaxNx && packed) {
      b = (w > kHash2HalfMaxW ? kBinBig : kBinHalf) + wedge_bin((int32_t)w) - kHashBins;
    } else if (w > 0) {
      b = kBinRest;
      if (w >= 16384 && nx < (1 << 26)) {
        const long long span = (long long)hub_cpw(nx) * tab;
        const long long blocks = ((long long)(h - (vgid ? gbase[vgid[h]] : 0)) + span - 1) / span;
        if (w >= blocks * (nx > 1024 ? nx : 1024)) {
          b = -1;
          hubs[atomicAdd(hist + kCBins, 1)] = {h, nx, w};
        }
      }
    }
    bin[k] = b;
    hw[k] = (int32_t)min(w, (long long)0x7fffffff);
    if (b >= 0) atomicAdd(&s_hist[b], 1);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kCBins; i += 256)
    if (s_hist[i]) atomicAdd(hist + i, s_hist[i]);
}

__global__ void __launch_bounds__(1024) k_cscatter(int32_t n_units, const int32_t* __restrict__ units,
                                                   const int32_t* __restrict__ bin, const int32_t* __restrict__ hw,
                                                   int32_t* __restrict__ cursor, int32_t n_hubs, int32_t n_hashed,
                                                   int32_t* __restrict__ cunits, int32_t* __restrict__ chash_w) {
  bin_vertices<kCBins, true>(
      n_units, cursor, [&](int32_t k) { return bin[k]; },
      [&](int32_t at, int32_t k) {
        cunits[n_hubs + at] = units[k];
        if (at < n_hashed) chash_w[at] = hw[k];
      });
}

// DevGraph::hpos: a row of CTAs per graph, thread per (row, bound).
__global__ void k_hub_pos(const HubGeom* __restrict__ geom, const HubSeg* __restrict__ seg,
                          const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int32_t* __restrict__ pos) {
  const HubGeom ge = geom[blockIdx.y];
  if (ge.nseg == 0) return;
  const int64_t per = ge.nseg + 1, total = (int64_t)(ge.end - ge.xmin) * per;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = ge.xmin + (int32_t)(t / per), k = (int32_t)(t % per);
    const int32_t id = k < ge.nseg ? seg[ge.seg + k].lo : seg[ge.seg + k - 1].hi;
    pos[ge.pos + t] = lower_bound_i32(ci, rp[x], rp[x + 1], id);
  }
}

// Bit rows of the graph, in both layouts (zeroed before): warp per row.
__global__ void k_bits(int32_t n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                       uint32_t* __restrict__ bits, uint32_t* __restrict__ bits_t) {
  const int lane = threadIdx.x & 31, W = (n + 31) / 32;
  const int x = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (x >= n) return;
  for (int32_t p = rp[x] + lane; p < rp[x + 1]; p += 32) {
    const int32_t y = ci[p];
    const uint32_t b = 1u << (y & 31);
    atomicOr(&bits[(size_t)x * W + (y >> 5)], b);
    atomicOr(&bits_t[(size_t)(y >> 5) * n + x], b);
  }
}

// Smallest slot whose reverse was not found (rev[p] == p): the input is not
// symmetric exactly when there is one.
__global__ void k_first_unreversed(int64_t nnz, const int32_t* __restrict__ rev, int32_t* __restrict__ first) {
  int32_t best = 0x7fffffff;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x)
    if (rev[p] == (int32_t)p) best = min(best, (int32_t)p);
  for (int o = 16; o; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
  if ((threadIdx.x & 31) == 0 && best != 0x7fffffff) atomicMin(first, best);
}

// ---- exclusive scan of int32 (totals fit int32) ----
__global__ void k_scan_tile_sums(int32_t n, const int32_t* __restrict__ in, int32_t* __restrict__ sums) {
  __shared__ int32_t ws[8];
  int32_t base = blockIdx.x * kScanTile;
  int32_t s = 0;
  for (int i = threadIdx.x; i < kScanTile; i += blockDim.x) {
    int32_t k = base + i;
    if (k < n) s += in[k];
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int32_t t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
    sums[blockIdx.x] = t;
  }
}

// single block: exclusive scan of the tile sums in place
__global__ void k_scan_sums(int32_t nb, int32_t* __restrict__ sums) {
  __shared__ int32_t ws[32];
  __shared__ int32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int32_t base = 0; base < nb; base += blockDim.x) {
    int32_t k = base + threadIdx.x;
    int32_t v = k < nb ? sums[k] : 0;
    int32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
      int32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
      int32_t t = lane < (int)(blockDim.x >> 5) ? ws[lane] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += y;
      }
      ws[lane] = t;
    }
    __syncthreads();
    int32_t pre = (w > 0 ? ws[w - 1] : 0) + x - v + carry;
    if (k < nb) sums[k] = pre;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = pre + v;
    __syncthreads();
  }
}

// out[k] = exclusive prefix, out[n] = total
__global__ void k_scan_tiles(int32_t n, const int32_t* __restrict__ in,
                             const int32_t* __restrict__ sums, int32_t* __restrict__ out) {
  __shared__ int32_t ws[8];
  const int per = kScanTile / 256;  // 8 consecutive elements per thread
  int32_t base = blockIdx.x * kScanTile + threadIdx.x * per;
  int32_t v[per];
  int32_t t = 0;
  for (int i = 0; i < per; ++i) {
    int32_t k = base + i;
    v[i] = k < n ? in[k] : 0;
    t += v[i];
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t x = t;
  for (int o = 1; o < 32; o <<= 1) {
    int32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    int32_t s = lane < 8 ? ws[lane] : 0;
    for (int o = 1; o < 8; o <<= 1) {
      int32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    if (lane < 8) ws[lane] = s;
  }
  __syncthreads();
  int32_t run = sums[blockIdx.x] + (w > 0 ? ws[w - 1] : 0) + x - t;
  for (int i = 0; i < per; ++i) {
    int32_t k = base + i;
    if (k < n) out[k] = run;
    run += v[i];
    if (k == n - 1) out[n] = run;
  }
}

int grid_for(int64_t work, int block) {
  int64_t g = (work + block - 1) / block;
  if (g < 1) g = 1;
  if (g > 65535LL * 16) g = 65535LL * 16;
  return (int)g;
}

}  // namespace

int order_key() {
  static int v = [] {
    const char* e = getenv("GC_ORDER");
    if (!e) return 0;
    if (!strcmp(e, "deg")) return 1;
    if (!strcmp(e, "none")) return 2;
    return 0;
  }();
  return v;
}

gc_status exclusive_scan(int32_t n, const int32_t* in, int32_t* out, cudaStream_t s) {
  if (n == 0) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int32_t), s);
    return e == cudaSuccess ? GC_OK : cuda_fail(e, "scan memset");
  }
  int32_t nb = (n + kScanTile - 1) / kScanTile;
  int32_t* sums = nullptr;
  cudaError_t e = pool_alloc(&sums, sizeof(int32_t) * nb, s);
  if (e != cudaSuccess) return cuda_fail(e, "scan alloc");
  k_scan_tile_sums<<<nb, 256, 0, s>>>(n, in, sums);
  k_scan_sums<<<1, 1024, 0, s>>>(nb, sums);
  k_scan_tiles<<<nb, 256, 0, s>>>(n, in, sums, out);
  e = cudaGetLastError();
  cudaFreeAsync(sums, s);
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "scan launch");
}

// Words of the hub kernel's count block (see kHubTabDefault).
int hub_tab_words() {
  static int v = [] {
    const char* e = getenv("GC_HUB_TAB_WORDS");
    const int x = e ? atoi(e) : kHubTabDefault;
    return (x >= 4096 && x <= kHeavyTab && x % 1024 == 0) ? x : kHubTabDefault;
  }();
  return v;
}

// Jobs per CTA of the hub kernel the hub units are cut into (environment
// GC_HUB_JOBS_PER_CTA, 0 .. 64, default 1; 0 keeps one job per hub), read
// once per process. With 1, only a hub that costs more than a whole CTA's
// share of the work is cut: every job looks at all lower neighbours of its hub,
// and heaviest-first stealing already balances hubs below that size (on R-MAT
// scale 22 the CTAs' lifetimes differ by 0.1 %).
static int hub_jobs_per_cta() {
  static int v = [] {
    const char* e = getenv("GC_HUB_JOBS_PER_CTA");
    const int x = e ? atoi(e) : 1;
    return x < 0 ? 0 : (x > 64 ? 64 : x);
  }();
  return v;
}

gc_status classify_c_units(int32_t n, const int32_t* d_rp, const int32_t* d_ci, const RankInfo& rank, PrepBuffers* p,
                           cudaStream_t s) {
  const int32_t nu = p->n_units;
  cudaError_t e = pool_alloc(&p->cunits, sizeof(int32_t) * (nu > 0 ? nu : 1), s);
  if (e != cudaSuccess) return cuda_fail(e, "alloc cunits");
  p->n_cheavy = 0;
  p->n_chash = 0;
  p->n_chash_big = 0;
  p->n_chash_mid = 0;
  p->n_chash2 = 0;
  p->n_chash2_big = 0;
  p->n_cunits = nu;
  int32_t largest = 0;
  for (int32_t gi = 0; gi < rank.G; ++gi) largest = std::max(largest, rank.gn[gi]);
  auto graph_of = [&](int32_t h) {
    return (size_t)(std::upper_bound(rank.gbase, rank.gbase + rank.G, h) - rank.gbase) - 1;
  };
  if (largest <= kSmemTableMax || nu == 0) {
    e = nu > 0 ? cudaMemcpyAsync(p->cunits, p->units, sizeof(int32_t) * nu, cudaMemcpyDeviceToDevice, s) : cudaSuccess;
    return e == cudaSuccess ? GC_OK : cuda_fail(e, "copy cunits");
  }
  const long long tab = hub_tab_words();
  const int sms = count_grid_size() / kCtasPerSm;
  HubUnit* d_hubs = nullptr;  // room for every unit; then the bins, the wedges and the histogram
  std::vector<HubUnit> heavy;
  int32_t hist[kCBins + 1];
  const size_t nu1 = (size_t)nu;
  e = pool_alloc(&d_hubs, sizeof(HubUnit) * nu1 + sizeof(int32_t) * (2 * nu1 + kCBins + 1), s);
  if (e != cudaSuccess) return cuda_fail(e, "classify pass-C units");
  int32_t* d_bin = reinterpret_cast<int32_t*>(d_hubs + nu1);
  int32_t *d_w = d_bin + nu1, *d_hist = d_w + nu1;
  e = cudaMemsetAsync(d_hist, 0, sizeof(hist), s);
  if (e == cudaSuccess) {
    k_cwork<<<std::min(grid_for((int64_t)nu * 32, 256), 8 * sms), 256, 0, s>>>(
        nu, p->units, d_rp, d_ci, p->rev, rank.d_vgid, rank.d_gbase, (int32_t)tab, largest <= kHash2MaxN, d_bin, d_w,
        d_hist, d_hubs);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(hist, d_hist, sizeof(hist), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  // hub units heaviest first, then the hashed units, the packed-key hash units
  // of the whole and of half tables, each by bins heaviest first, and the rest
  if (e == cudaSuccess) {
    int32_t cursor[kCBins], at = 0;
    auto place = [&](int b) {
      cursor[b] = at;
      at += hist[b];
    };
    for (int b = kHashBins - 1; b >= 0; --b) {
      place(b);
      if (b == wedge_bin(kHashMidW + 1)) p->n_chash_mid = at;
      if (b == wedge_bin(kHashSmallW + 1)) p->n_chash_big = at;
    }
    p->n_chash = at;
    for (int b = kBinRest - 1; b >= kBinBig; --b) place(b);
    p->n_chash2_big = at - p->n_chash;
    for (int b = kBinBig - 1; b >= kBinHalf; --b) place(b);
    p->n_chash2 = at - p->n_chash;
    const int32_t n_hashed = at;
    place(kBinRest);
    p->n_cheavy = hist[kCBins];
    p->n_cunits = p->n_cheavy + at;
    try {
      heavy.resize((size_t)p->n_cheavy);
    } catch (...) {
      e = cudaErrorMemoryAllocation;
    }
    if (n_hashed > 0 && e == cudaSuccess) e = pool_alloc(&p->chash_w, sizeof(int32_t) * (size_t)n_hashed, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_hist, cursor, sizeof(cursor), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && at > 0) {
      k_cscatter<<<std::min(grid_for(nu, 1024), 2 * sms), 1024, 0, s>>>(nu, p->units, d_bin, d_w, d_hist, p->n_cheavy,
                                                                        n_hashed, p->cunits, p->chash_w);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess && !heavy.empty())
      e = cudaMemcpyAsync(heavy.data(), d_hubs, sizeof(HubUnit) * heavy.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  cudaFreeAsync(d_hubs, s);
  if (e != cudaSuccess) return cuda_fail(e, "classify pass-C units");
  std::sort(heavy.begin(), heavy.end(),
            [](const HubUnit& a, const HubUnit& b) { return a.w != b.w ? a.w > b.w : a.h < b.h; });
  // The hub kernel's o-range (see HubSeg): per graph, segment by segment, the
  // counter width that reaches furthest (the wider one at equal reach): to the
  // end of the ids whose degree fits it, or of the block. A block is closed when
  // less than a sixteenth is left. Every (neighbour, segment) costs a look at
  // the row, so that a graph whose ids all fit one block of 16-bit counters
  // gets one segment, not one per degree class.
  std::vector<HubSeg> segs;
  std::vector<HubGeom> geom;
  int64_t n_pos = 0;
  if (!heavy.empty()) {
    for (int32_t gi = 0; gi < rank.G; ++gi) {
      const int32_t* ob = rank.obound + (size_t)gi * kOBounds;
      const int32_t end = rank.gbase[gi] + rank.gn[gi];
      HubGeom ge = {(int32_t)segs.size(), 0, end, end, n_pos};
      int32_t word = 0;
      for (int32_t lo = ob[0], hi; lo < end; lo = hi) {
        int lg = 0;
        hi = lo;
        for (int l = 0; l < kOBounds; ++l) {
          const int32_t fits = l == 0 ? end : ob[kOBounds - l];  // ids whose degree fits 32 >> l bits
          const int32_t to = (int32_t)std::min<int64_t>(fits, lo + ((tab - word) << l));
          if (to > hi) {
            hi = to;
            lg = l;
          }
        }
        segs.push_back({lo, hi, word, (int16_t)lg, 0});
        word += (hi - lo + (1 << lg) - 1) >> lg;
        if (tab - word < tab / 16 || hi == end) {
          segs.back().last = 1;
          word = 0;
        }
      }
      ge.nseg = (int32_t)segs.size() - ge.seg;
      if (ge.nseg > 0) {
        // rows of at least max(32, bounds) entries: the last ids
        const int32_t least = std::max(32, ge.nseg + 1);
        int32_t a = rank.gbase[gi], b = end;
        while (a < b) {
          const int32_t mid = a + (b - a) / 2;
          if (rank.rp[mid + 1] - rank.rp[mid] < least) a = mid + 1; else b = mid;
        }
        ge.xmin = a;
        n_pos += (int64_t)(end - a) * (ge.nseg + 1);
      }
      geom.push_back(ge);
    }
  }
  // Hub units cut into jobs of consecutive o-ranges (the finer granularity of
  // Sec. 4.4: one hub's work spread over several CTAs), so that the heaviest
  // hubs do not end as one SM's serial tail. A unit's cost is estimated as
  // its wedges plus kSweepCost per (lower neighbour, segment) sweep; a unit is
  // cut into about cost / target jobs, target = total cost over jobs_per_cta
  // x the hub kernel's CTAs (GC_HUB_JOBS_PER_CTA, default 1; 0: one job per
  // hub), at ids that split the entries of its o-range's rows evenly (an o
  // is met about in proportion to its degree). A job looks at every lower
  // neighbour, so it keeps at least kJobWedges wedges and eight for each of
  // them. Jobs are taken heaviest first.
  std::vector<int4> jobs;
  if (!heavy.empty()) {
    constexpr double kSweepCost = 4.0;
    constexpr long long kJobWedges = 8192;
    const int per_cta = hub_jobs_per_cta();
    auto geom_of = [&](int32_t h) -> const HubGeom& {
      return geom[graph_of(h)];
    };
    auto seg_of = [&](const HubGeom& ge, int32_t id) {  // the segment holding id (the last one past the end)
      int32_t k = ge.seg;
      while (k + 1 < ge.seg + ge.nseg && segs[(size_t)k].hi <= id) ++k;
      return k;
    };
    std::vector<double> cost(heavy.size());
    double total = 0;
    for (size_t i = 0; i < heavy.size(); ++i) {
      const HubUnit& k = heavy[i];
      const HubGeom& ge = geom_of(k.h);
      cost[i] = (double)k.w + kSweepCost * (double)k.nx * (double)(seg_of(ge, k.h) - ge.seg + 1);
      total += cost[i];
    }
    const double target = per_cta > 0 ? total / ((double)(count_grid_size() / kCtasPerSm) * per_cta) : 0.0;
    std::vector<std::pair<double, int4>> cj;
    for (size_t i = 0; i < heavy.size(); ++i) {
      const int32_t h = heavy[i].h;
      const HubGeom& ge = geom_of(h);
      const int32_t lo = ge.nseg > 0 ? std::min(segs[(size_t)ge.seg].lo, h) : h;
      long long J = target > 0 ? (long long)std::ceil(cost[i] / target) : 1;
      J = std::max(1LL, std::min(J, heavy[i].w / std::max(kJobWedges, 8LL * heavy[i].nx)));
      int32_t from = lo;
      for (long long j = 1; j <= J; ++j) {
        const long long upto = rank.rp[lo] + (long long)(rank.rp[h] - rank.rp[lo]) * j / J;
        const int32_t to =
            j == J ? h : (int32_t)(std::upper_bound(rank.rp + lo, rank.rp + h, (int32_t)upto) - rank.rp) - 1;
        if (to <= from && (j < J || from > lo)) continue;  // nothing in this share (a hub keeps at least one job)
        cj.push_back({cost[i] / (double)J, make_int4((int)i, from, to, 2 * seg_of(ge, from) + (from == lo))});
        from = to;
      }
    }
    std::stable_sort(cj.begin(), cj.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
    jobs.reserve(cj.size());
    for (auto& c : cj) jobs.push_back(c.second);
    // device copies: the geometry and the segments in one block, and the rows' positions
    const size_t gb = sizeof(HubGeom) * geom.size(), sb = sizeof(HubSeg) * segs.size();
    e = pool_alloc(&p->hgeom, gb + sb + sizeof(HubSeg), s);
    if (e == cudaSuccess) p->hseg = reinterpret_cast<HubSeg*>(p->hgeom + geom.size());
    if (e == cudaSuccess) e = cudaMemcpyAsync(p->hgeom, geom.data(), gb, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && sb) e = cudaMemcpyAsync(p->hseg, segs.data(), sb, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = pool_alloc(&p->hpos, sizeof(int32_t) * (size_t)(n_pos > 0 ? n_pos : 1), s);
    int64_t widest = 0;
    for (const HubGeom& ge : geom) widest = std::max(widest, (int64_t)(ge.end - ge.xmin) * (ge.nseg + 1));
    for (size_t g0 = 0; g0 < geom.size() && widest > 0 && e == cudaSuccess; g0 += 32768) {
      const dim3 grid((unsigned)std::min(grid_for(widest, 256), 4096), (unsigned)std::min<size_t>(32768, geom.size() - g0));
      k_hub_pos<<<grid, 256, 0, s>>>(p->hgeom + g0, p->hseg, d_rp, d_ci, p->hpos);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_fail(e, "hub layout");
  }
  p->n_cjobs = (int32_t)jobs.size();
  if (!jobs.empty()) {
    e = pool_alloc(&p->cjobs, sizeof(int4) * jobs.size(), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(p->cjobs, jobs.data(), sizeof(int4) * jobs.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return cuda_fail(e, "hub jobs");
  }
  std::vector<int32_t> out;
  out.reserve(heavy.size());
  for (const HubUnit& k : heavy) out.push_back(k.h);
  if (!out.empty()) e = cudaMemcpyAsync(p->cunits, out.data(), sizeof(int32_t) * out.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "copy cunits");
}

gc_status first_unreversed_slot(int64_t nnz, const int32_t* d_rev, int32_t* out, cudaStream_t s) {
  *out = -1;
  if (nnz <= 0) return GC_OK;
  int32_t* d = nullptr;
  cudaError_t e = pool_alloc(&d, sizeof(int32_t), s);
  const int32_t init = 0x7fffffff;
  int32_t h = init;
  if (e == cudaSuccess) e = cudaMemcpyAsync(d, &init, sizeof(int32_t), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    k_first_unreversed<<<grid_for(nnz, 256) > 4096 ? 4096 : grid_for(nnz, 256), 256, 0, s>>>(nnz, d_rev, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (d) cudaFreeAsync(d, s);
  if (e != cudaSuccess) return cuda_fail(e, "symmetry check");
  *out = h == init ? -1 : h;
  return GC_OK;
}

gc_status build_bits(int32_t n, const int32_t* d_rp, const int32_t* d_ci, PrepBuffers* p, cudaStream_t s) {
  const size_t words = (size_t)n * (size_t)((n + 31) / 32);
  cudaError_t e = pool_alloc(&p->bits, sizeof(uint32_t) * 2 * words, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(p->bits, 0, sizeof(uint32_t) * 2 * words, s);
  if (e != cudaSuccess) return cuda_fail(e, "bit rows");
  p->bits_t = p->bits + words;
  k_bits<<<grid_for((int64_t)n * 32, 256), 256, 0, s>>>(n, d_rp, d_ci, p->bits, p->bits_t);
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "k_bits");
}

void free_prep(PrepBuffers* p, cudaStream_t s) {
  if (p->bits) cudaFreeAsync(p->bits, s);
  if (p->deg) cudaFreeAsync(p->deg, s);
  if (p->eid) cudaFreeAsync(p->eid, s);
  if (p->uv) cudaFreeAsync(p->uv, s);
  if (p->out_ptr) cudaFreeAsync(p->out_ptr, s);
  if (p->out_idx) cudaFreeAsync(p->out_idx, s);
  if (p->units) cudaFreeAsync(p->units, s);
  if (p->rev) cudaFreeAsync(p->rev, s);
  if (p->ocsr) cudaFreeAsync(p->ocsr, s);
  if (p->e2o) cudaFreeAsync(p->e2o, s);
  if (p->kunits) cudaFreeAsync(p->kunits, s);
  if (p->cunits) cudaFreeAsync(p->cunits, s);
  if (p->cjobs) cudaFreeAsync(p->cjobs, s);
  if (p->chash_w) cudaFreeAsync(p->chash_w, s);
  if (p->hgeom) cudaFreeAsync(p->hgeom, s);
  if (p->hpos) cudaFreeAsync(p->hpos, s);
  *p = PrepBuffers();
}

gc_status prepare_graph(int32_t n, int32_t m, const int32_t* d_rp, const int32_t* d_ci, int32_t* d_eid,
                        const int32_t* d_perm, const RankInfo& rank, PrepBuffers* out, cudaStream_t s) {
  PrepBuffers P;
  P.eid = d_eid;
  int32_t *out_cnt = nullptr, *dmax = nullptr, *hist = nullptr;
  gc_status st = GC_OK;
  cudaError_t e = cudaSuccess;
  const int64_t nnz = 2 * (int64_t)m;
#define GC_TRY(call, what)                 \
  do {                                     \
    e = (call);                            \
    if (e != cudaSuccess) {                \
      st = cuda_fail(e, what);             \
      goto fail;                           \
    }                                      \
  } while (0)
  GC_TRY(pool_alloc(&P.deg, sizeof(int32_t) * (n > 0 ? n : 1), s), "alloc deg");
  GC_TRY(pool_alloc(&P.rev, sizeof(int32_t) * (nnz > 0 ? nnz : 1), s), "alloc rev");
  GC_TRY(pool_alloc(&P.out_ptr, sizeof(int32_t) * ((int64_t)n + 1), s), "alloc out_ptr");
  GC_TRY(pool_alloc(&P.out_idx, sizeof(int32_t) * (m > 0 ? m : 1), s), "alloc out_idx");
  GC_TRY(pool_alloc(&P.units, sizeof(int32_t) * (n > 0 ? n : 1), s), "alloc units");
  GC_TRY(pool_alloc(&P.ocsr, sizeof(int32_t) * (m > 0 ? m : 1), s), "alloc ocsr");
  if (d_eid) {
    GC_TRY(pool_alloc(&P.uv, sizeof(int32_t) * (nnz > 0 ? nnz : 1), s), "alloc uv");
    GC_TRY(pool_alloc(&P.e2o, sizeof(int32_t) * (m > 0 ? m : 1), s), "alloc e2o");
    GC_TRY(cudaMemsetAsync(P.e2o, 0, sizeof(int32_t) * (m > 0 ? m : 1), s), "memset e2o");  // in range whatever the input
  }
  GC_TRY(pool_alloc(&P.kunits, sizeof(int32_t) * (n > 0 ? n : 1), s), "alloc kunits");
  GC_TRY(pool_alloc(&out_cnt, sizeof(int32_t) * (n > 0 ? n : 1), s), "alloc out_cnt");
  // [0] max degree, [1..64] v-group bins, [65] max out-degree, [66..97] pass-K
  // bins, [98..101] the sums of d^2 and of k (d - k), 64 bits each
  GC_TRY(pool_alloc(&dmax, sizeof(int32_t) * 102, s), "alloc dmax");
  hist = dmax + 1;
  GC_TRY(cudaMemsetAsync(dmax, 0, sizeof(int32_t) * 102, s), "memset");
  if (n > 0) {
    const int blocks = std::min(grid_for(n, 256), 8 * (count_grid_size() / kCtasPerSm));
    const int bin_blocks = std::min(grid_for(n, 1024), 2 * (count_grid_size() / kCtasPerSm));
    k_deg_out<<<blocks, 256, 0, s>>>(n, d_rp, d_ci, P.deg, out_cnt, dmax, dmax + 65,
                                  reinterpret_cast<unsigned long long*>(dmax + 98));
    GC_TRY(cudaGetLastError(), "k_deg_out");
    if ((st = exclusive_scan(n, out_cnt, P.out_ptr, s)) != GC_OK) goto fail;
    k_rev_init<<<grid_for(nnz, 256), 256, 0, s>>>(nnz, P.rev);
    GC_TRY(cudaGetLastError(), "k_rev_init");
    k_edges<<<grid_for((int64_t)n * 32, 256), 256, 0, s>>>(n, m, d_rp, d_ci, P.out_ptr, P.eid, P.out_idx, P.ocsr,
                                                            P.rev, P.e2o, d_perm);
    GC_TRY(cudaGetLastError(), "k_edges");
    if (d_eid) {
      k_uv_perm<<<grid_for((int64_t)n * 32, 256), 256, 0, s>>>(n, d_rp, d_ci, P.eid, d_perm, P.uv);
      GC_TRY(cudaGetLastError(), "k_uv_perm");
    }
    k_bin_units<false><<<bin_blocks, 1024, 0, s>>>(n, P.deg, out_cnt, hist, nullptr, order_key());
    GC_TRY(cudaGetLastError(), "k_bin_units");
    k_bin_kunits<false><<<bin_blocks, 1024, 0, s>>>(n, out_cnt, dmax + 66, nullptr);
    GC_TRY(cudaGetLastError(), "k_bin_kunits");
    {
      int32_t h[102];
      GC_TRY(cudaMemcpyAsync(h, dmax, sizeof(h), cudaMemcpyDeviceToHost, s), "copy hist");
      GC_TRY(cudaStreamSynchronize(s), "sync hist");
      P.dmax = h[0];
      P.kmax = h[65];
      uint64_t sums[2];
      std::memcpy(sums, h + 98, sizeof(sums));
      int64_t n2 = 0;
      int32_t largest = 0;
      for (int32_t gi = 0; gi < rank.G; ++gi) {
        n2 += (int64_t)rank.gn[gi] * rank.gn[gi];
        largest = std::max(largest, rank.gn[gi]);
      }
      P.route = small_route(largest, rank.G, n2, m, P.kmax, (double)sums[0], (double)sums[1]);
      {  // pass-K units, largest bin first; tier boundaries at k = 1024, 512, 256, 32
        int32_t kc[32];
        int32_t acc = 0;
        for (int b = 31; b >= 0; --b) {
          if (b == 10) P.ktier_off[kTier1024] = acc;
          if (b == 9) P.ktier_off[kTier512] = acc;
          if (b == 8) P.ktier_off[kTier256] = acc;
          if (b == 5) P.ktier_off[kTier32] = acc;
          kc[b] = acc;
          acc += h[66 + b];
        }
        P.ktier_off[kTierGlobal] = 0;
        P.ktier_off[kNumTiers] = acc;
        GC_TRY(cudaMemcpyAsync(dmax + 66, kc, sizeof(kc), cudaMemcpyHostToDevice, s), "copy k cursors");
        k_bin_kunits<true><<<bin_blocks, 1024, 0, s>>>(n, out_cnt, dmax + 66, P.kunits);
        GC_TRY(cudaGetLastError(), "k_bin_kunits");
      }
      int32_t cur[64];
      int32_t acc = 0;
      for (int b = 63; b >= 0; --b) {  // heaviest bin first
        cur[b] = acc;
        acc += h[1 + b];
      }
      P.n_units = acc;
      GC_TRY(cudaMemcpyAsync(hist, cur, sizeof(cur), cudaMemcpyHostToDevice, s), "copy cursors");
      k_bin_units<true><<<bin_blocks, 1024, 0, s>>>(n, P.deg, out_cnt, hist, P.units, order_key());
      GC_TRY(cudaGetLastError(), "k_bin_units");
    }
  } else {
    GC_TRY(cudaMemsetAsync(P.out_ptr, 0, sizeof(int32_t), s), "memset out_ptr");
  }
  try {
    st = classify_c_units(n, d_rp, d_ci, rank, &P, s);
  } catch (...) {
    st = no_memory();
  }
  if (st != GC_OK) goto fail;
  cudaFreeAsync(out_cnt, s);
  cudaFreeAsync(dmax, s);
  *out = P;
  return GC_OK;
fail:
  cudaStreamSynchronize(s);
  if (out_cnt) cudaFreeAsync(out_cnt, s);
  if (dmax) cudaFreeAsync(dmax, s);
  free_prep(&P, s);
  return st;
#undef GC_TRY
}

}  // namespace gc
