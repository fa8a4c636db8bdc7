// gc_noalloc.cu -- a triangle-count entry point that allocates no memory.
//
// Callers that own a fixed memory arena, or that run where a device
// allocation may not happen at all (inside another allocator's callback,
// under a hard budget that forbids growth), cannot use gc_graph_upload: it
// allocates the CSR copy, the preparation arrays and the per-CTA tables. This
// entry point is a variant of the triangle step (Alg. 1) that works directly
// on the caller's device CSR and writes the caller's device output. Its only
// scratch lives in a file-scope __device__ array of 32 MiB that every GPU
// loading the library holds until the process exits. Graphs with more than
// kNoAllocMaxN vertices are rejected.
//
// tri[p] of the slot p = (x, y) is the number of entries of row y that are in
// row x. In a simple symmetric graph the slots of both directions agree, so
// each edge is counted once, at its end of higher (degree, id): the entries of
// the shorter row are looked up in a set of the longer one. That is
// sum min(d_x, d_y) lookups over the edges, where looking up row y in a bitmap
// of row x for every slot, in global memory, took sum d^2 (Chung-Lu, 100 003
// vertices, 1 000 003 edges, exponent 2.3: 2.2e9 lookups and 7.9 ms for a
// pass, 0.45 ms now: 37 us k_rows, 318 k_tri, whose warps wait at barriers for the
// longest chain of loads among them, 66 k_tri_reverse, which waits on loads).
// Up to kOneN vertices one kernel does it all, a CTA per row (k_tri_one). Above,
// five launches, each waiting for the one before:
//   k_rows   marks the rows that break the CSR rules (not strictly ascending,
//            a column out of range, a self-loop) and lists the long rows
//   k_tri    the slots (x, y), y below x in (degree, id): a CTA per part of a
//            long row with a bitmap of the vertices in shared memory, then a
//            warp per other row with a hash of at most 128 entries (or 256)
//   k_tri_reverse   the other slots, from the reverse slot (a binary search);
//            slots without one, or with an end whose row breaks the rules, are
//            marked
//   k_tri_marked    the marked slots by the definition, with a bitmap per CTA in
//            the scratch array (nothing to do for a valid graph)
// Up to kPickN vertices k_pick, in the place of the clearing, picks either.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "gc_deal.h"
#include "gc_internal.h"

namespace gc {
namespace {

constexpr int32_t kNoAllocMaxN = 1 << 20;              // vertices
constexpr int kNoAllocWords = kNoAllocMaxN / 32;       // 32-bit words of a bitmap of the vertices
constexpr int kNoAllocCtas = 192;                      // CTAs of k_tri_marked, one bitmap each
constexpr int kNoAllocBlock = 512;
// Scratch layout, in 32-bit words: counters, a bit per row that breaks the
// CSR rules, the list of long rows, the bitmaps of k_tri_marked.
enum { kCurLong = 0, kNumLong, kCurShort, kNumMarked, kOneKernel, kNumCounters };
constexpr size_t kOffBad = 32;
constexpr size_t kOffLong = kOffBad + kNoAllocWords;
constexpr size_t kOffMaps = (size_t)2 * kNoAllocMaxN;
constexpr size_t kScratchWords = kOffMaps + (size_t)kNoAllocCtas * kNoAllocWords;  // 32 MiB
static_assert(kScratchWords * 4 == (size_t)32 << 20, "scratch size");

// Up to this many vertices, the bitmap and the warps' hashes leave room for four
// CTAs an SM, and one kernel takes the long rows and then the short ones.
constexpr int32_t kBothMaxN = 1 << 17;
// Up to this many, the bitmap leaves room for four CTAs of 512 threads an SM beside
// the 13 KB that every CTA takes; beyond, fewer fit, of 1024 threads.
constexpr int32_t kFourMaxN = 358400;

// Slots of a long row that a warp takes at a time: the runs of that many lower
// neighbours are a warp's chain of loads. Graphs of fewer entries have fewer
// warps' worth of slots, and there the longest chain is the kernel's time
// (Chung-Lu, exponent 2.3, a pass with one split of 32 slots for all sizes, with
// this one, and of the bitmap in global memory: 20 000 edges 260, 67, 68 us;
// 50 000 edges 283, 84, 143; 100 000 edges 286, 96, 341; 10^6 edges 611, 504, 7690).
__device__ __forceinline__ int window_of(int64_t nnz) { return nnz < (1 << 18) ? 8 : nnz < (1 << 20) ? 16 : 32; }
// Rows of at most this many entries are a warp's (d^2 / 128 steps at most); a
// longer one is a CTA's, in parts of a window per warp. Where large bitmaps leave
// one or two CTAs an SM, a part's barriers and chains of loads are hidden badly and
// rows up to 256 entries are a warp's, in graphs of many (10^6 vertices, up to 128
// and 256 entries: 7700 complete graphs of 135, 52 and 23 ms; 5000 of 200, 75 and
// 44; Chung-Lu, 5e7 edges, exponent 4, 23.1 and 18.5; 10^7, 2.1, 5.40 and 5.44; at
// 300 000 vertices, 1.5e7 edges, 5.21 and 5.60).
__device__ __forceinline__ int short_row(int32_t n, int64_t nnz) {
  return n > kFourMaxN && nnz >= (1 << 24) ? 256 : 4 * window_of(nnz);
}
// (from 2^28 entries larger ones, so that their list holds all of them: 1700
// complete graphs of 600, which it did not hold, 1163 ms, now 392)
__device__ __forceinline__ int part_of(int64_t nnz) {
  return nnz < (1 << 28) ? kNoAllocBlock / 32 * window_of(nnz) : 2048;
}
constexpr int kShortRow = 128;              // the longest short row up to kFourMaxN vertices
constexpr int kShortSlots = 2 * kShortRow;  // its hash, at most half full
constexpr int kShortWords = kShortSlots + kShortRow;  // a warp's hash and filter
constexpr int kMidSlots = 2 * 256, kMidWords = kMidSlots + kShortRow;  // beyond
constexpr int kTriBlock = 256;
constexpr int kMaxHeavy = 512;              // heavy runs of a part that its warps share
// A lower neighbour's row of this many entries is shared by all warps, as one
// alone would be the last to end (R-MAT scale 18, rows from 512, 1024, 2048
// entries: 1.99, 1.71, 1.68 ms; 950 complete graphs of 1100: 1368, 1367, 1211).
constexpr int kHeavyRun = 2048;
constexpr uint32_t kMaxParts = (uint32_t)(kOffMaps - kOffLong);  // list entries: x (20 bits) and the part above
constexpr uint32_t kNoPart = 0xffffffffu;
// Up to kOneN vertices, k_tri_one does the whole step; up to kPickN, it or the
// kernels of larger graphs, picked from the degrees on the device.
constexpr int32_t kOneN = 1024, kPickN = 4096;

static __device__ __align__(256) uint32_t g_noalloc_scratch[kScratchWords];

// Device address of g_noalloc_scratch, looked up once per device ordinal and
// kept for the life of the process: this assumes the device's primary context
// (the one the CUDA runtime uses) and no cudaDeviceReset in between, after
// which the cached address would name memory of a context that is gone.
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
uint32_t* g_noalloc_ptr[kMaxDevices] = {};
int g_noalloc_sms[kMaxDevices] = {};  // SMs of the device, with the address

// Up to kCloseN vertices the kernels of a call follow each other closely: a kernel
// lets the next one be launched as soon as all its CTAs run, and the next one waits
// here until the previous is complete and its writes can be seen. Beyond, the next
// kernel's waiting CTAs cost more than the gap (Chung-Lu, 100 003 vertices, 10^6
// edges: 495 us, closely 509; R-MAT scale 13 111 and 106; a cycle of 4097 76 and 65).
constexpr int32_t kCloseN = 1 << 14;
__device__ __forceinline__ void after_previous() {
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
}
template <class... Params, class... Args>
cudaError_t launch_after(void (*kernel)(Params...), int grid, int block, size_t smem, cudaStream_t s, int32_t n,
                         Args... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = n <= kCloseN;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, n, args...);
}

__device__ __forceinline__ bool row_bad(const uint32_t* scratch, int32_t x) {
  return (scratch[kOffBad + (x >> 5)] >> (x & 31)) & 1u;
}

// Thread per slot: rows with a column out of range, a self-loop or two entries
// out of order; thread per row: the long rows, in parts. (A warp
// per row would walk the longest rows alone: 0.4 ms for one of 25 000 entries.)
__global__ void __launch_bounds__(kTriBlock) k_rows(int32_t n, const int32_t* __restrict__ rp,
                                                    const int32_t* __restrict__ ci, uint32_t* __restrict__ scratch) {
  after_previous();
  if (scratch[kOneKernel]) return;
  const int lane = threadIdx.x & 31;
  const int64_t t0 = (int64_t)blockIdx.x * kTriBlock + threadIdx.x, threads = (int64_t)gridDim.x * kTriBlock;
  const int64_t nnz = rp[n];
  const int32_t part = part_of(nnz), longest_short = short_row(n, nnz);
  for (int64_t x = t0; x < n; x += threads) {
    const int32_t d = rp[x + 1] - rp[x];
    if (d <= longest_short) continue;
    if (d > n || d > nnz) {  // more entries than vertices
      atomicOr(scratch + kOffBad + (x >> 5), 1u << (x & 31));
      continue;
    }
    const uint32_t parts = (uint32_t)((d + part - 1) / part);  // at most 4096, as d <= min(n, nnz)
    const uint32_t at = atomicAdd(scratch + kNumLong, parts);
    // else by k_tri_marked: more parts than the list holds (only beyond 2.08e9
    // entries), or a last part of the last vertex that would read as kNoPart
    const bool fits = at + parts <= kMaxParts && !((uint32_t)x == 0xfffffu && parts == 4096u);
    if (!fits) atomicOr(scratch + kOffBad + (x >> 5), 1u << (x & 31));
    for (uint32_t k = 0; k < parts && at + k < kMaxParts; ++k)
      scratch[kOffLong + at + k] = fits ? (uint32_t)x | (k << 20) : kNoPart;
  }
  for (int64_t p = t0; p - lane < nnz; p += threads) {
    const int32_t p0 = (int32_t)(p - lane), p_last = (int32_t)min((int64_t)p0 + 31, nnz - 1);
    const int32_t q = (int32_t)min(p, nnz - 1);
    const int32_t x = row_of_slot(n, rp, p0, q, p_last);
    const int32_t y = ci[q];
    if ((uint32_t)y >= (uint32_t)n || y == x || (q > rp[x] && ci[q - 1] >= y))
      atomicOr(scratch + kOffBad + (x >> 5), 1u << (x & 31));
  }
}

// The lower neighbours of x in one window of 32 slots of its row, which starts at
// b: the lane's is the k-th, if below end, and whether it is counted here (both
// rows follow the rules, and y is below x in (degree, id)); its row [yb, yb + L).
// Places in a row are counted from its start all through these kernels: a slot,
// which may be up to 2^31 - 2, plus a step or another slot would not fit 32 bits.
__device__ __forceinline__ void lower_slot(int32_t n, const int32_t* rp, const int32_t* ci, const uint32_t* scratch,
                                           int32_t x, int32_t dx, int32_t b, int32_t k, int32_t end, int32_t& yb,
                                           int32_t& L, bool& mine) {
  yb = L = 0;
  mine = false;
  if (k >= end) return;
  const int32_t y = ci[b + k];
  if ((uint32_t)y >= (uint32_t)n || row_bad(scratch, y)) return;
  yb = rp[y];
  const int32_t dy = rp[y + 1] - yb;
  mine = dy < dx || (dy == dx && y < x);
  L = mine ? dy : 0;
}

// Counts, for 32 runs laid end to end over the lanes (lane l's run is [yb, yb +
// L)), the entries for which `in` holds, per run in cnt[32] (the warp's).
template <class In>
__device__ __forceinline__ void count_runs(const int32_t* __restrict__ ci, int32_t yb, int32_t L, int32_t* cnt, int lane,
                                           In in) {
  int32_t incl = L;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  const int32_t total = __shfl_sync(0xffffffffu, incl, 31), base = yb - (incl - L);
  for (int32_t k0 = 0; k0 < total; k0 += 128) {  // four windows of loads in flight
    int32_t w[4], own[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int32_t k = k0 + 32 * j + lane;
      int r = 0;  // the run of position k: how many runs end at or before it
#pragma unroll
      for (int step = 16; step; step >>= 1)
        if (__shfl_sync(0xffffffffu, incl, r + step - 1) <= k) r += step;
      own[j] = r;
      const int32_t b = __shfl_sync(0xffffffffu, base, r);
      w[j] = k < total ? ci[b + k] : -1;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (w[j] >= 0 && in(w[j])) atomicAdd(&cnt[own[j]], 1);
  }
}

// The same with the runs of kLongRun entries or more read by the whole warp, one
// after the other, at a third of the instructions an entry (k_tri: 1000 complete
// graphs of 500, 659 ms with all runs laid end to end, now 271; K_300, 3400 of
// them, 376 and 130). `in` takes any number.
constexpr int32_t kLongRun = 64;
template <class In>
__device__ __forceinline__ void count_runs_long(const int32_t* __restrict__ ci, int32_t yb, int32_t L, int32_t* cnt,
                                                int lane, In in) {
  count_runs(ci, yb, L < kLongRun ? L : 0, cnt, lane, in);
  unsigned lm = __ballot_sync(0xffffffffu, L >= kLongRun);
  while (lm) {
    const int src = __ffs(lm) - 1;
    lm &= lm - 1u;
    const int32_t* row = ci + __shfl_sync(0xffffffffu, yb, src);
    const uint32_t len = (uint32_t)__shfl_sync(0xffffffffu, L, src);
    uint32_t c = 0;
    for (uint32_t q = lane; q < len; q += 128) {
      int32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) w[j] = q + 32 * j < len ? row[q + 32 * j] : -1;
#pragma unroll
      for (int j = 0; j < 4; ++j) c += in(w[j]);
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == src) cnt[lane] = (int32_t)c;  // its own: count_runs left it 0
  }
}

// The whole step in one kernel: CTA per row x, a bitmap of it in shared memory; a
// window of its slots per warp, whose short rows are read end to end over the
// lanes and whose long ones (kLongRun entries) by the whole warp. Every slot by
// the definition, so that no row's order matters: sum d^2 lookups, where the
// kernels below take sum min(d_x, d_y) but four more launches. A call with the
// read-back of row_ptr[n] around it (about 30 us), one kernel / the others:
// G(64, 0.3) 40 / 71 us, G(1000, 0.02) 43 / 82, K_1000 687 / 795, K(200, 800)
// 161 / 151; the others' 71 is 66 since they follow each other closely.
constexpr int kOneBlock = 256;
__global__ void __launch_bounds__(kOneBlock) k_tri_one(int32_t n, const int32_t* __restrict__ rp,
                                                       const int32_t* __restrict__ ci, int32_t* __restrict__ tri,
                                                       const uint32_t* scratch /* null: not picked */) {
  constexpr int kW = kOneBlock / 32;
  __shared__ uint32_t bm[kPickN / 32];
  if (scratch) {  // else the call's only kernel: what follows it is the caller's
    after_previous();
    if (!scratch[kOneKernel]) return;
  }
  __shared__ int32_t s_cnt[kW][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int32_t* cnt = s_cnt[warp];
  auto in = [&](int32_t w) -> bool { return (uint32_t)w < (uint32_t)n && ((bm[w >> 5] >> (w & 31)) & 1u); };
  for (int32_t x = blockIdx.x; x < n; x += gridDim.x) {
    const int32_t b = rp[x];
    const uint32_t d = (uint32_t)(rp[x + 1] - b);
    if (d == 0u) continue;
    __syncthreads();  // the previous row's lookups
    for (int i = threadIdx.x; i < (n + 31) / 32; i += kOneBlock) bm[i] = 0u;
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < d; k += kOneBlock) {
      const int32_t w = ci[b + k];
      if ((uint32_t)w < (uint32_t)n) atomicOr(&bm[w >> 5], 1u << (w & 31));
    }
    __syncthreads();
    const uint32_t window = min(32u, (d + kW - 1) / kW);  // slots a warp takes at a time
    for (uint32_t k0 = warp * window; k0 < d; k0 += kW * window) {
      const bool mine = lane < window && k0 + lane < d;
      int32_t yb = 0, L = 0;
      if (mine) {
        const int32_t y = ci[b + k0 + lane];
        if ((uint32_t)y < (uint32_t)n) {
          yb = rp[y];
          L = rp[y + 1] - yb;
        }
      }
      cnt[lane] = 0;
      __syncwarp();
      count_runs_long(ci, yb, L, cnt, lane, in);
      __syncwarp();
      if (mine) tri[b + k0 + lane] = cnt[lane];
      __syncwarp();
    }
  }
}

// One CTA, in the place of clearing the counters and the bad-row bits: does that,
// and picks k_tri_one or the kernels after it: the first where sum d^2 is small
// anyway, or the degrees are about equal (E[d^2] <= 1.25 E[d]^2), where sum min(d)
// saves little. k_tri_one / the others: G(3000, 0.1) 298 / 382 us, G(2000, 0.01)
// 46 / 70, Chung-Lu 4000 / 10 000 63 / 72, star of 4000 71 / 69, Chung-Lu 4000 /
// 60 000 130 / 97, K(100, 3900) 978 / 193, G(2048, 0.7) 2810 / 2469.
__global__ void __launch_bounds__(1024) k_pick(int32_t n, const int32_t* __restrict__ rp, uint32_t* __restrict__ scratch) {
  __shared__ double s_d2[32];
  cudaTriggerProgrammaticLaunchCompletion();
  double d2 = 0;
  for (int32_t x = threadIdx.x; x < n; x += 1024) {
    const double d = (double)(rp[x + 1] - rp[x]);
    d2 += d * d;
  }
  for (int32_t i = threadIdx.x; i < (int32_t)kOffBad + (n + 31) / 32; i += 1024)
    if (i != kOneKernel) scratch[i] = 0u;
  for (int o = 16; o; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
  if ((threadIdx.x & 31) == 0) s_d2[threadIdx.x >> 5] = d2;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) d2 += s_d2[w];
    const double nnz = (double)rp[n];
    scratch[kOneKernel] = d2 <= 8e6 || (d2 <= 2e9 && d2 * n <= 1.25 * nnz * nnz);
  }
}

// Warp per row of up to short_row() entries: its entries in an open-addressing
// hash (twice the slots), behind a filter of 16 bits a hash slot (8 where the row
// has more than 128 entries).
__device__ __forceinline__ void short_rows(int32_t n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                           int32_t* __restrict__ tri, uint32_t* __restrict__ scratch, int32_t* key,
                                           uint32_t* filt, int32_t* cnt, int lane) {
  const int32_t longest = short_row(n, rp[n]);
  // rows taken at a time: eight where every warp gets many
  const int32_t take = min(8, max(1, n / (int32_t)(gridDim.x * (kNoAllocBlock / 32))));
  for (;;) {
    int32_t x0 = 0;
    if (lane == 0) x0 = (int32_t)atomicAdd(scratch + kCurShort, (uint32_t)take);
    x0 = __shfl_sync(0xffffffffu, x0, 0);
    if (x0 >= n) break;
    for (int32_t x = x0; x < min(x0 + take, n); ++x) {
      const int32_t b = rp[x], d = rp[x + 1] - b;
      if (d > longest || d == 0 || row_bad(scratch, x)) continue;  // warp-uniform
      int bits = 5;
      while ((1 << bits) < 2 * d) ++bits;  // at most log2(kShortSlots), or of kMidSlots
      const uint32_t mask = (1u << bits) - 1u;
      const int fbits = min(bits + 4, 12);  // kShortRow words at most
      for (int i = lane; i <= (int)mask; i += 32) key[i] = -1;
      for (int i = lane; i < (1 << fbits) / 32; i += 32) filt[i] = 0u;
      __syncwarp();
      for (int32_t k = lane; k < d; k += 32) {
        const int32_t y = ci[b + k];
        const uint32_t hy = (uint32_t)y * 0x9E3779B1u;
        uint32_t s = hy >> (32 - bits);
        while (atomicCAS(&key[s], -1, y) != -1) s = (s + 1) & mask;  // rows ascend: no y twice, half full
        const uint32_t f = ((uint32_t)y * 0x85EBCA6Bu) >> (32 - fbits);
        atomicOr(&filt[f >> 5], 1u << (f & 31));
      }
      __syncwarp();
      for (int32_t k0 = 0; k0 < d; k0 += 32) {
        int32_t yb, L;
        bool mine;
        lower_slot(n, rp, ci, scratch, x, d, b, k0 + lane, d, yb, L, mine);
        cnt[lane] = 0;
        __syncwarp();
        count_runs(ci, yb, L, cnt, lane, [&](int32_t w) -> bool {
          const uint32_t f = ((uint32_t)w * 0x85EBCA6Bu) >> (32 - fbits);
          if (!((filt[f >> 5] >> (f & 31)) & 1u)) return false;
          uint32_t s = ((uint32_t)w * 0x9E3779B1u) >> (32 - bits);
          for (;;) {
            const int32_t k = key[s];
            if (k == w) return true;
            if (k == -1) return false;
            s = (s + 1) & mask;
          }
        });
        __syncwarp();
        if (mine) tri[b + k0 + lane] = cnt[lane];
        __syncwarp();
      }
    }
  }
}

// CTA per part of a long row: a bitmap of the n vertices in shared memory with
// the whole row; the warps take windows of the part's slots, and leave the
// long rows of lower neighbours to a list that all warps then read together
// (the heaviest neighbours are often next to each other, and one warp alone
// took 0.9 ms for them).
template <int kThreads>
__device__ __forceinline__ void long_parts(int32_t n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                           int32_t* __restrict__ tri, uint32_t* __restrict__ scratch,
                                           uint32_t* bm /* (n + 31) / 32 words */, int32_t* cnt) {
  __shared__ uint32_t s_x;
  __shared__ int32_t s_next, s_heavy;
  __shared__ int32_t s_hp[kMaxHeavy], s_hb[kMaxHeavy], s_hl[kMaxHeavy], s_hc[kMaxHeavy];  // slots, rows, counts
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nnz = rp[n];
  const int32_t slots = part_of(nnz);
  const uint32_t n_long = min(scratch[kNumLong], kMaxParts);
  // Bounds are checked although the listed rows follow the rules: calls that
  // overlap on the GPU share the scratch array, and may then list rows and miss
  // marks of each other's graphs.
  auto in = [&](int32_t w) -> bool { return (uint32_t)w < (uint32_t)n && ((bm[w >> 5] >> (w & 31)) & 1u); };
  for (int32_t i = threadIdx.x; i < (n + 31) / 32; i += kThreads) bm[i] = 0u;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t k, v;
      do {
        k = atomicAdd(scratch + kCurLong, 1u);
        v = k < n_long ? scratch[kOffLong + k] : kNoPart;
      } while (k < n_long && v == kNoPart);
      s_x = v;
    }
    __syncthreads();
    if (s_x == kNoPart) break;
    const int32_t x = (int32_t)(s_x & 0xfffffu), part = (int32_t)(s_x >> 20);
    if (x >= n || row_bad(scratch, x)) continue;
    const int32_t b = rp[x], d = rp[x + 1] - b;
    const int32_t start = min(d, part * slots), end = min(d, start + slots);  // at most 4096 parts of 128 to 2048 slots
    const int32_t window = min(32, (end - start + kThreads / 32 - 1) / (kThreads / 32));  // some for every warp
    if (threadIdx.x == 0) {
      s_next = start;
      s_heavy = 0;
    }
    for (int32_t k = threadIdx.x; k < d; k += kThreads) {
      const int32_t y = ci[b + k];
      if ((uint32_t)y < (uint32_t)n) atomicOr(&bm[y >> 5], 1u << (y & 31));
    }
    __syncthreads();
    for (;;) {
      int32_t k0 = 0;
      if (lane == 0) k0 = atomicAdd(&s_next, window);
      k0 = __shfl_sync(0xffffffffu, k0, 0);
      if (k0 >= end) break;
      int32_t yb, L;
      bool mine;
      lower_slot(n, rp, ci, scratch, x, d, b, k0 + lane, min(end, k0 + window), yb, L, mine);
      if (L >= kHeavyRun) {
        const int32_t k = atomicAdd(&s_heavy, 1);
        if (k < kMaxHeavy) {  // else this warp's
          s_hp[k] = b + k0 + lane;
          s_hb[k] = yb;
          s_hl[k] = L;
          s_hc[k] = 0;
          L = 0;
          mine = false;
        }
      }
      cnt[lane] = 0;
      __syncwarp();
      count_runs_long(ci, yb, L, cnt, lane, in);
      __syncwarp();
      if (mine) tri[b + k0 + lane] = cnt[lane];
      __syncwarp();
    }
    __syncthreads();
    const int32_t heavy = min(s_heavy, kMaxHeavy);
    int32_t before = 0;  // their pieces of 128 entries go round the warps
    for (int32_t k = 0; k < heavy; ++k) {
      const int32_t *row = ci + s_hb[k], len = s_hl[k];
      int32_t c = 0;
      for (int32_t q0 = 128 * ((warp - before) & (kThreads / 32 - 1)); q0 < len; q0 += 128 * (kThreads / 32)) {
        int32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = q0 + 32 * j + lane < len ? row[q0 + 32 * j + lane] : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) c += in(w[j]);
      }
      before += (len + 127) >> 7;
      c = (int32_t)__reduce_add_sync(0xffffffffu, (unsigned)c);
      if (lane == 0 && c) atomicAdd(&s_hc[k], c);
    }
    __syncthreads();
    for (int32_t k = threadIdx.x; k < heavy; k += kThreads) tri[s_hp[k]] = s_hc[k];
    for (int32_t k = threadIdx.x; k < d; k += kThreads) {
      const int32_t y = ci[b + k];
      if ((uint32_t)y < (uint32_t)n) bm[y >> 5] = 0u;
    }
  }
}

// Both, or one of them (which: bit 0 long rows, bit 1 short ones), with the
// bitmap and the warps' hashes in dynamic shared memory.
template <int kThreads>
__global__ void __launch_bounds__(kThreads, 2048 / kThreads)
    k_tri(int32_t n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, int32_t* __restrict__ tri,
          uint32_t* __restrict__ scratch, int which) {
  extern __shared__ uint32_t s_dyn[];
  __shared__ int32_t s_cnt[kThreads / 32][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  after_previous();
  if (scratch[kOneKernel]) return;
  uint32_t* tables = s_dyn;
  if (which & 1) {
    long_parts<kThreads>(n, rp, ci, tri, scratch, s_dyn, s_cnt[warp]);
    tables += (n + 31) / 32;
  }
  if (which & 2) {
    uint32_t* mine = tables + warp * (n > kFourMaxN ? kMidWords : kShortWords);
    short_rows(n, rp, ci, tri, scratch, reinterpret_cast<int32_t*>(mine),
               mine + (n > kFourMaxN ? kMidSlots : kShortSlots), s_cnt[warp], lane);
  }
}

// The slots (x, y) with y above x: the value of the reverse slot. Thread per
// slot.
__global__ void __launch_bounds__(kTriBlock) k_tri_reverse(int32_t n, const int32_t* __restrict__ rp,
                                                           const int32_t* __restrict__ ci, int32_t* __restrict__ tri,
                                                           uint32_t* __restrict__ scratch) {
  after_previous();
  if (scratch[kOneKernel]) return;
  const int lane = threadIdx.x & 31;
  const int64_t nnz = rp[n], threads = (int64_t)gridDim.x * kTriBlock;
  bool marked = false;
  for (int64_t p = (int64_t)blockIdx.x * kTriBlock + threadIdx.x; p - lane < nnz; p += threads) {
    const int32_t p0 = (int32_t)(p - lane), p_last = (int32_t)min((int64_t)p0 + 31, nnz - 1);
    const int32_t q = (int32_t)min(p, nnz - 1);
    const int32_t x = row_of_slot(n, rp, p0, q, p_last);
    if (p >= nnz) continue;
    const int32_t y = ci[q], dx = rp[x + 1] - rp[x];
    bool found = false;
    if ((uint32_t)y < (uint32_t)n && !row_bad(scratch, x) && !row_bad(scratch, y)) {
      const int32_t yb = rp[y], ye = rp[y + 1], dy = ye - yb;
      if (dy < dx || (dy == dx && y < x)) continue;  // counted at this slot
      int32_t lo = yb, hi = ye;
      while (lo < hi) {
        const int32_t mid = lo + ((hi - lo) >> 1);
        if (ci[mid] < x) lo = mid + 1; else hi = mid;
      }
      found = lo < ye && ci[lo] == x;
      if (found) tri[q] = tri[lo];
    }
    if (!found) {
      tri[q] = -1;
      marked = true;
    }
  }
  if (marked) atomicAdd(scratch + kNumMarked, 1u);
}

// The marked slots, by the definition: the row's columns marked in the CTA's
// bitmap, the row of each marked slot's column looked up in it by one warp, the
// bitmap cleared again. A column outside [0, n) is skipped; its own slot gets 0.
__global__ void __launch_bounds__(kNoAllocBlock) k_tri_marked(int32_t n, const int32_t* __restrict__ rp,
                                                              const int32_t* __restrict__ ci, int32_t* __restrict__ tri,
                                                              uint32_t* __restrict__ scratch) {
  cudaGridDependencySynchronize();
  if (scratch[kNumMarked] == 0u) return;
  uint32_t* bm = scratch + kOffMaps + (size_t)blockIdx.x * kNoAllocWords;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int warps = kNoAllocBlock / 32;
  const int32_t words = (n + 31) / 32;  // the array keeps the previous call's contents: start from zero
  for (int32_t i = threadIdx.x; i < words; i += kNoAllocBlock) bm[i] = 0u;
  __syncthreads();
  for (int32_t x = blockIdx.x; x < n; x += gridDim.x) {
    const int32_t xb = rp[x];
    const uint32_t d = (uint32_t)(rp[x + 1] - xb);
    bool any = false;
    for (uint32_t k = threadIdx.x; k < d; k += kNoAllocBlock) any |= tri[xb + k] == -1;
    if (!__syncthreads_or(any)) continue;
    for (uint32_t k = threadIdx.x; k < d; k += kNoAllocBlock) {
      const int32_t w = ci[xb + k];
      if ((uint32_t)w < (uint32_t)n) atomicOr(&bm[w >> 5], 1u << (w & 31));
    }
    __syncthreads();
    for (uint32_t k = warp; k < d; k += warps) {
      if (tri[xb + k] != -1) continue;
      const int32_t y = ci[xb + k];
      int c = 0;
      if ((uint32_t)y < (uint32_t)n)
        for (uint32_t q = lane; q < (uint32_t)(rp[y + 1] - rp[y]); q += 32) {
          const int32_t w = ci[rp[y] + q];
          if ((uint32_t)w < (uint32_t)n) c += (bm[w >> 5] >> (w & 31)) & 1u;
        }
      c = (int)__reduce_add_sync(0xffffffffu, (unsigned)c);
      if (lane == 0) tri[xb + k] = c;
    }
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < d; k += kNoAllocBlock) {
      const int32_t w = ci[xb + k];
      if ((uint32_t)w < (uint32_t)n) bm[w >> 5] = 0u;
    }
    __syncthreads();
  }
}

}  // namespace
}  // namespace gc

using namespace gc;

extern "C" gc_status gc_edge_triangles_noalloc(int32_t n, const int32_t* row_ptr, const int32_t* col_idx,
                                               int32_t* tri_out, void* stream) try {
  if (n < 0 || (n > 0 && (!row_ptr || !col_idx || !tri_out))) {
    set_error("gc_edge_triangles_noalloc: bad arguments");
    return GC_ERR_ARG;
  }
  if (n > kNoAllocMaxN) {
    set_error("gc_edge_triangles_noalloc: n = " + std::to_string(n) + " exceeds the fixed scratch limit of " +
              std::to_string(kNoAllocMaxN) + " vertices");
    return GC_ERR_OVERFLOW;
  }
  if (n == 0) return GC_OK;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("gc_edge_triangles_noalloc: device index out of range");
    return GC_ERR_ARG;
  }
  uint32_t* scratch = nullptr;
  int sms = 0;
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      // first call on this device (the current one): resolve the host-side
      // symbol to the device address of the array
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress");
      if ((e = cudaDeviceGetAttribute(&g_noalloc_sms[dev], cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return cuda_fail(e, "cudaDeviceGetAttribute");
      for (auto kernel : {k_tri<kNoAllocBlock>, k_tri<2 * kNoAllocBlock>})
        if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kNoAllocWords * 4)) !=
            cudaSuccess)
          return cuda_fail(e, "k_tri");
      g_noalloc_ptr[dev] = static_cast<uint32_t*>(p);
    }
    scratch = g_noalloc_ptr[dev];
    sms = g_noalloc_sms[dev];
  }
  cudaStream_t s = (cudaStream_t)stream;
  if (n <= kOneN) {
    k_tri_one<<<std::min(n, sms * 8), kOneBlock, 0, s>>>(n, row_ptr, col_idx, tri_out, nullptr);
    e = cudaGetLastError();
    return e == cudaSuccess ? GC_OK : cuda_fail(e, "gc_edge_triangles_noalloc");
  }
  const size_t bitmap = sizeof(uint32_t) * (size_t)((n + 31) / 32);
  const size_t tables = sizeof(uint32_t) * (n > kFourMaxN ? kMidWords : kShortWords) * (kNoAllocBlock / 32);
  const int grid = sms * 8;  // 2048 threads an SM; the number of slots is on the device only
  // the counters and the bad-row bits cleared; then each kernel is launched while
  // the one before it runs, and waits for it (after_previous)
  if (n <= kPickN) {
    k_pick<<<1, 1024, 0, s>>>(n, row_ptr, scratch);
    launch_after(k_tri_one, std::min(n, grid), kOneBlock, 0, s, n, row_ptr, col_idx, tri_out, scratch);
  } else if ((e = cudaMemsetAsync(scratch, 0, sizeof(uint32_t) * (kOffBad + (size_t)((n + 31) / 32)), s)) !=
             cudaSuccess) {
    return cuda_fail(e, "zero counters");
  }
  launch_after(k_rows, grid, kTriBlock, 0, s, n, row_ptr, col_idx, scratch);
  auto tri = [&](int which, int per_sm, int block, size_t smem) {
    launch_after(block == kNoAllocBlock ? k_tri<kNoAllocBlock> : k_tri<2 * kNoAllocBlock>, sms * per_sm, block, smem, s,
                 n, row_ptr, col_idx, tri_out, scratch, which);
  };
  // CTAs an SM: four (2048 threads) while the bitmaps leave room for them in
  // 227 KB, beside the 11 KB that every CTA takes; with larger bitmaps fewer, of
  // twice the threads (R-MAT scale 20: 20.7 ms with 512, 15.2 with 1024)
  if (n <= kBothMaxN) {
    tri(3, 4, kNoAllocBlock, bitmap + tables);
  } else {
    if (n <= kFourMaxN) tri(1, 4, kNoAllocBlock, bitmap);
    else tri(1, bitmap + (15 << 10) <= (size_t)227 * 512 ? 2 : 1, 2 * kNoAllocBlock, bitmap);
    tri(2, 4, kNoAllocBlock, tables);
  }
  launch_after(k_tri_reverse, grid, kTriBlock, 0, s, n, row_ptr, col_idx, tri_out, scratch);
  launch_after(k_tri_marked, kNoAllocCtas, kNoAllocBlock, 0, s, n, row_ptr, col_idx, tri_out, scratch);
  e = cudaGetLastError();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "gc_edge_triangles_noalloc");
} catch (...) {
  return no_memory();
}
