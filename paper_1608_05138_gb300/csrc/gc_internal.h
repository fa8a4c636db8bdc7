// gc_internal.h -- shared declarations of libgc's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <functional>
#include <memory>
#include <string>
#include <vector>

#include "../../include/gc.h"

namespace gc {

typedef unsigned __int128 u128;

// The o-range of the hub kernel of pass C, laid out once per ranked graph: a
// vertex of degree 1 closes no 4-cycle, and a count of o never exceeds d_o, so
// ids, which ascend by degree, split at these degrees into classes of 2-, 4-,
// 8-, 16- and 32-bit counters (kOBoundDeg[k] is where class k starts).
constexpr int kOBounds = 5;
constexpr int kOBoundDeg[kOBounds] = {2, 4, 16, 256, 65536};
// One segment: ids [lo, hi), 2^lg counters to a 32-bit word, from word `word`
// of the count block. Consecutive segments share a block until one is `last`.
struct HubSeg {
  int32_t lo, hi, word;
  int16_t lg, last;
};
// Segments of one graph, and the places of its segment bounds in the rows:
// row x >= xmin (the rows of at least 32 entries and of more entries than
// bounds) has, for its k-th segment, its first slot of id >= lo, and the slot
// past the last segment: hpos[pos + (x - xmin) * (nseg + 1) + k].
struct HubGeom {
  int32_t seg, nseg, xmin, end;
  int64_t pos;
};

// Device view of a (possibly multi-graph) CSR. A batch of graphs is counted
// as their disjoint union: vertices of graph g occupy the global id range
// [gbase[g], gbase[g] + gn[g]); per-edge x3/x7/x10 of a disjoint union equal
// those of each component, while n and m in the per-edge columns and the sums
// are taken per graph.
struct DevGraph {
  int32_t n;               // vertices in total
  int32_t m;               // undirected edges in total
  const int32_t* rp;       // [n + 1] row pointers (global ids)
  const int32_t* ci;       // [2m] column ids (global ids), rows ascending
  const int32_t* deg;      // [n]
  const int32_t* eid;      // [2m] slot -> edge id
  const int32_t* out_ptr;  // [n + 1] degree-oriented out-lists (P3 orientation)
  const int32_t* out_idx;  // [m] ascending ids within each list; position = out-slot
  const int32_t* ocsr;     // [m] out-slot -> CSR slot of the same direction (row of the owner)
  const int32_t* e2o;      // [m] edge id -> out-slot
  const int32_t* rev;      // [2m] slot of (y, x) for the slot of (x, y)
  int32_t G;               // graphs in the union (>= 1)
  const int32_t* vgid;     // [n] graph of each vertex, or nullptr when G == 1
  const int32_t* gbase;    // [G] first global vertex id of each graph
  const int32_t* gn;       // [G] vertices of each graph
  const int64_t* gm;       // [G] edges of each graph
  int32_t table_n;         // max gn[g]: size of one Psi table
  const uint32_t* bits;    // kRouteDense (small_route()): bit rows [n][(n + 31) / 32], and the same by word
  const uint32_t* bits_t;  // [(n + 31) / 32][n]; else nullptr
  const HubGeom* hgeom;    // ranked: [G] (nullptr when the graph has no hub units)
  const HubSeg* hseg;
  const int32_t* hpos;
  int32_t n_long;          // one graph: rows of more than 4096 entries, the last ids
};

// Pass K (4-cliques and cross terms by lowest vertex) runs in tiers by the
// out-degree k of the lowest vertex: the local bitmatrix of out(a) lives in
// shared memory up to k = 1024 and in a per-CTA global buffer above.
// Units with k <= 32 are done by one warp each, with the rows in registers.
enum KTier { kTierGlobal = 0, kTier1024, kTier512, kTier256, kTier32, kNumTiers };
constexpr int kTierCap[kNumTiers] = {0, 1024, 512, 256, 32};

// Counting configuration chosen on the host.
struct CountArgs {
  const int32_t* units;    // pass C: v-groups (high endpoints), heaviest bin first
  int32_t n_units;
  const int32_t* cunits;   // pass C: hub units (blocked kernel), hashed units, then the others
  int32_t n_cheavy;        // hub units of pass C (cunits[0 .. n_cheavy))
  const int32_t* chash_w;  // wedges of the hashed units cunits[n_cheavy .. n_cheavy + n_chash + n_chash2)
  int32_t n_chash;
  int32_t n_chash_mid;     // hashed units of more than kHashMidW wedges (the first of them)
  int32_t n_chash_big;     // hashed units of more than kHashSmallW wedges (the first of them)
  int32_t n_chash2;        // units of the packed-key hash tier, after the hashed units
  int32_t n_chash2_big;    // of them, units of more than kHash2HalfMaxW wedges (the first)
  const int4* cjobs;       // pass C hub kernel: jobs (hub index into cunits, o-range [y, z), twice the
                           // segment of y, + 1 for the hub's first job), heaviest first
  int32_t n_cjobs;
  int32_t hub_tab;         // pass C hub kernel: words of the count block (hub_tab_words())
  const int32_t* kunits;   // pass K: lowest vertices a with |out(a)| >= 2, tiers in KTier order
  int32_t ktier_off[kNumTiers + 1];  // tier t = kunits[ktier_off[t] .. ktier_off[t + 1])
  int32_t* cursor;         // work-stealing cursors (device ints, zeroed before each launch)
  uint32_t* tables;        // global Psi tables (grid x table_n) or nullptr (shared memory)
  int32_t* trio;           // [m] |T| by out-slot (pass T)
  unsigned long long* P;   // [2m] per slot: 4-cycles through its edge counted at that slot
                           // (pass C, zeroed before); an edge's count = sum of its two slots
  unsigned long long* xc;    // [m][2] per out-slot: 4-cliques through the edge, and the sum over T of
                             // (|T_(a,u)| + |T_(a,v)| - 2) (pass K); side by side, so that the two
                             // atomics of an edge land in one 32-byte sector
  uint32_t* x7d;           // dense graphs: [n][n] 4-cliques through the edge (lower, higher); else nullptr
  unsigned char* kbuf;     // global-tier per-CTA buffers (kbuf_ctas x kbuf_stride bytes)
  size_t kbuf_stride;
  int32_t kbuf_ctas;
  int32_t kbuf_cap;        // largest k the global tier holds
  int2* hitbuf;            // passes T/K: per-CTA lists of the edges of H_a; tier t (tiers run side by side) has
                           // hit_ctas[t] lists of hit_cap[t] entries from hit_off[t]
  int64_t hit_off[kNumTiers];
  int32_t hit_cap[kNumTiers];
  int32_t hit_ctas[kNumTiers];
  // Edges of every H_a, recorded by pass T for pass K (nullptr: not kept):
  // entry = ((i << 16) | j, out-slot of (b_i, b_j)); unit ui (index into
  // kunits) has tl_cnt[ui] entries from tl_off[ui], or tl_cnt[ui] = -1.
  int2* tlist;
  long long tlist_cap;
  unsigned long long* tlist_fill;
  long long* tl_off;
  int32_t* tl_cnt;
  unsigned long long* dsum;  // [m] per out-slot: sum over T of d_w (pass T, per-edge induced counts only)
  uint64_t* per_edge;      // [m][13] device pointer or nullptr
  bool per_edge_host;      // per_edge maps pinned host memory
  unsigned long long* csum;  // [G][13][2] 128-bit unrestricted counts (lo, hi)
  int32_t* status;         // device status word (0 = ok)
  unsigned long long* work;  // [kNumWork] work counters of this count
};

// Work counters (units the kernels processed; bench.py turns them into
// algorithmic bytes).
enum Work {
  kWorkTMembers = 0,   // pass T: sum over units of |out(a)|
  kWorkCWedge,         // pass C: wedges h-x-o
  kWorkKMembers,       // pass K: sum over units of |out(a)|
  kWorkKScan,          // pass K: out-list entries scanned to build the local graphs
  kWorkKLocalEdges,    // pass K: local edges = triangles (each once)
  kWorkKWords,         // pass K: bitmatrix words ANDed (local edges x row words)
  kWorkFinishEdges,    // finish: edges written
  kWorkLaunches,       // kernels launched by the count (counted on the host)
  kWorkCHeavyWedge,    // pass C: wedges of the hub units (blocked kernel)
  kWorkCBlocks,        // pass C: lower neighbours swept, summed over the blocks of the hub units
  kWorkTScan,          // pass T: out-list entries scanned
  kWorkTTriangles,     // pass T: triangles (each once)
  kWorkCHashWedge,     // pass C: wedges of the units counted in a shared-memory hash
  kWorkCHubJobs,       // pass C: jobs of the hub kernel (hub units cut into ranges of o-range blocks)
  kWorkCHubCtas,       // pass C: CTAs of the hub kernel
  kWorkCHubBusySum,    // pass C: sum over the hub kernel's CTAs of their lifetime (ns, %globaltimer)
  kWorkCHubBusyMax,    // pass C: the longest of those lifetimes (ns)
  kWorkCHash2Wedge,    // pass C: wedges of the units counted in the packed-key hash
  kNumWork
};

// Device status bits. kSpillOverflow: a unit outgrew what it was binned for
// (a pass-T/K tier, the hashed pass-C table); it cannot
// happen for a validated graph.
enum Status : int32_t { kOk = 0, kSpillOverflow = 1, kInexact = 2 };

constexpr int kBlock = 512;            // threads per CTA of pass C's vertex-indexed tables
constexpr int kCtasPerSm = 2;          // resident CTAs per SM of the persistent grids
constexpr int kWarps = kBlock / 32;
constexpr int kSmemTableMax = 4096;    // Psi tables up to this many vertices live in shared memory

// Phases timed with CUDA events.
enum Phase { kPhasePassT = 0, kPhasePassC, kPhasePassK, kPhaseFinish, kPhaseInduced, kPhaseDerive, kPhaseCopy,
             kNumPhases };

// Side streams of one count, kept by the library and lent to one count of a graph
// handle (or to one stream slot of a batch) at a time: kernels of a phase that do
// not depend on each other run side by side on `stream`, forked from the count's
// own stream by `start` and joined by `done`. A handle keeps none between its
// counts: a stream takes 0.57 MB of device memory and 13 us to make, and 1000 live
// handles with ten each took 5.7 GB and 0.5 ms longer for their first counts.
constexpr int kForkStreams = 10;
struct ForkSet {
  cudaStream_t stream[kForkStreams] = {};
  cudaEvent_t start = nullptr, done[kForkStreams] = {};
  int device = 0;
  int priority = 0;  // of its streams
};
// What a graph handle keeps: events that time the phases of its last count, and
// pinned memory that receives the results.
constexpr size_t kPinnedBytes = 1024;
struct CountTimers {
  cudaEvent_t begin[kNumPhases] = {}, end[kNumPhases] = {};
  unsigned char* pinned = nullptr;
};
ForkSet* fork_acquire(int device, int priority);  // of the current device; nullptr on failure (message set)
// Whether the stream belongs to a part of the GPU only (a green context): its
// count then stays on it, since side streams would be on the whole GPU.
bool on_part_of_gpu(cudaStream_t s);
void fork_release(ForkSet* f);   // its streams must be idle; nullptr is accepted
void fork_drain(ForkSet* f);     // waits for its streams (after a failed count, whose forks were not joined)

// Side streams of one fork: next() is a stream that starts where the main
// stream stood at the constructor, join() makes the main stream wait for all
// of them. Without a set everything stays on the main stream.
class Fork {
 public:
  Fork(cudaStream_t s, ForkSet* f, int first, int count) : s_(s), f_(f), first_(first), count_(count) {
    if (f_) e_ = cudaEventRecord(f_->start, s_);
  }
  cudaStream_t next() {
    if (!f_ || used_ >= count_ || e_ != cudaSuccess) return s_;
    cudaStream_t& t = f_->stream[first_ + used_];
    cudaEvent_t& d = f_->done[first_ + used_];
    if (!t) e_ = cudaStreamCreateWithPriority(&t, cudaStreamNonBlocking, f_->priority);  // on first use, and kept
    if (!d && e_ == cudaSuccess) e_ = cudaEventCreateWithFlags(&d, cudaEventDisableTiming);
    if (e_ == cudaSuccess) e_ = cudaStreamWaitEvent(t, f_->start, 0);
    if (e_ != cudaSuccess) return s_;  // join() reports it
    ++used_;
    return t;
  }
  cudaError_t join() {
    for (int k = 0; k < used_; ++k) {  // also after a failure: what was forked is waited for
      cudaError_t e = cudaEventRecord(f_->done[first_ + k], f_->stream[first_ + k]);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s_, f_->done[first_ + k], 0);
      if (e_ == cudaSuccess) e_ = e;
    }
    used_ = 0;
    return e_;
  }

 private:
  cudaStream_t s_;
  ForkSet* f_;
  int first_, count_, used_ = 0;
  cudaError_t e_ = cudaSuccess;
};

// Device scratch of one count (lazily grown; owned by a graph handle or by
// one batch launch).
struct Scratch {
  // one block, zeroed before every count: the results' head (misc: cursors and
  // status, work, fill, csum [G][13][2], x [G][17][2]), then trio, xc and P
  unsigned char* zero = nullptr;
  size_t zero_bytes = 0, head_bytes = 0;
  int32_t* misc = nullptr;             // [32]
  unsigned long long* work = nullptr;  // [kNumWork]
  unsigned long long* tl_fill = nullptr;
  unsigned long long* csum = nullptr;
  unsigned long long* x = nullptr;
  int32_t* trio = nullptr;           // [m]
  unsigned long long* xc = nullptr;  // [m][2]
  unsigned long long* P = nullptr;   // [2m]
  uint32_t* x7d = nullptr;           // [n][n] (dense graphs)
  uint32_t* tables = nullptr;        // count_grid_size() x table_n
  size_t tables_n = 0;
  unsigned char* kbuf = nullptr;     // pass K global tier
  size_t kbuf_stride = 0;
  int32_t kbuf_ctas = 0;
  int32_t kbuf_cap = 0;
  int2* hitbuf = nullptr;            // per-CTA H_a edge lists (see CountArgs)
  int64_t hit_off[kNumTiers] = {};
  int32_t hit_cap[kNumTiers] = {};
  int32_t hit_ctas[kNumTiers] = {};
  int2* tlist = nullptr;             // edges of all H_a, from pass T to pass K
  long long tlist_cap = 0;           // entries
  long long tlist_want = 0;          // triangles of the last count (or a first guess): the size to keep
  long long* tl_off = nullptr;       // [units of pass K]
  int32_t* tl_cnt = nullptr;
  int32_t tl_units = 0;
  int32_t launches = 0;              // kernels launched by the last run_count
  unsigned long long* dsum = nullptr;  // [m] per-edge induced counts: sum over T of d_w
  unsigned long long* vsum = nullptr;  // [n][2] per-edge induced counts: 2 x triangles, neighbour degrees
};
// Allocates the scratch of a union of G graphs with m edges, Psi tables of
// table_n vertices, largest out-degree kmax and pass-K tiers tier_off, and for
// a dense graph its vertices dense_n (stream-ordered).
gc_status scratch_init(Scratch* sc, int32_t m, int32_t table_n, int32_t kmax, const int32_t* tier_off, int32_t G,
                       int32_t dense_n, cudaStream_t s);
void scratch_free(Scratch* sc, cudaStream_t s);
// Size of pass T's edge lists for the first count of a whole graph with m
// edges: 32 m entries within the list budget (units past it scan again).
void scratch_guess_tlist(Scratch* sc, int64_t m);
// The whole count: passes T, C, K, finish, derive; the sums and X land in
// sc->csum and sc->x. Kernels that do not depend on each other run side by
// side on the set's streams, pass C beside passes T and K in graphs of fewer
// than kOverlapEdges edges (see run_count). Returns after the derive is queued
// (no host synchronisation).
struct KUnits {
  int32_t kmax;            // largest out-degree
  const int32_t* units;
  int32_t tier_off[kNumTiers + 1];
  const int32_t* cunits;   // pass C units: hubs, hashed units, the others
  int32_t n_cheavy;
  const int4* cjobs;       // hub jobs (see CountArgs)
  int32_t n_cjobs;
  const int32_t* chash_w;
  int32_t n_chash;
  int32_t n_chash_mid;
  int32_t n_chash_big;
  int32_t n_chash2;
  int32_t n_chash2_big;
  int32_t n_cunits;        // pass C units in all (units without wedges are left out)
  bool rows;               // the graph's route (small_route) is not kRoutePasses
};
// induced (optional): [m][10] rows of the per-edge induced counts of H_7..H_16
// (device pointer, or the device view of pinned host memory when
// induced_host), written after the finish.
gc_status run_count(const DevGraph& g, const int32_t* units, int32_t n_units, const KUnits& ku,
                    uint64_t* per_edge, Scratch* sc, cudaStream_t s, ForkSet* fs, CountTimers* tm,
                    bool per_edge_host = false, uint64_t* induced = nullptr, bool induced_host = false);

// How a graph, or a union of graphs, is counted: by passes T, C and K; from rows
// of common neighbours (run_rows) for graphs of at most kSmemTableMax vertices;
// or from those on bit rows (run_rows_dense), one graph of 64 to kDenseMaxN
// vertices with out-degrees up to kDenseMaxK.
enum SmallRoute { kRoutePasses = 0, kRouteRows, kRouteDense };
constexpr int kDenseMaxN = 2048;
constexpr int kDenseMaxK = 1024;
// n vertices of the largest of G graphs, n2 the sum of their n^2, m edges in
// all, kmax the largest out-degree, d2 = sum d^2, kd = sum k (d - k), the
// out-list entries that pass T scans. What the three routes cost (GB300, us a
// count with per-edge rows; passes / rows / dense):
//   rows read 2 d2 entries (1.1 us per 10^6), whatever they find; the passes'
//   work follows kd and the triangles. G(3000, 0.03), d2 2.5e7: 243 / 194;
//   Chung-Lu 4000 / 60 000 edges, 3.1e7: 360 / 309; 20 hubs joined to 4000
//   others, 3.2e8: 575 / 512; 200 hubs joined to 2000, 7.3e8: 526 / 1035;
//   K(500, 3500), 7.0e9: 2470 / 7828; G(4096, 0.1), 6.9e8: 1269 / 1569.
//   Above 2.5e8 they pay only where most of what they read are triangles, that is
//   in graphs as dense all over as G(n, 0.2), d2 = 6 kd there: G(3000, 0.3),
//   2.4e9: 5793 / 5503; G(4096, 0.3), 6.2e9: 19596 / 17803; Chung-Lu 4000 /
//   10^6, d2 = 8.7 kd: 2723 / 3318.
//   Without a vertex of two higher neighbours nothing is left for passes T and K:
//   star of 4000 leaves 324 / 412.
//   Bit rows cost n / 32 words a slot and bit of the counts, and a k x k matrix per
//   vertex whether it has edges or not: G(500, 0.3) 169 / 152 / 129, G(1000, 0.1)
//   169 / 138 / 150, G(1000, 0.3) 422 / 353 / 245, G(1500, 0.2) 483 / 457 / 409,
//   G(2000, 0.11) 342 / 341 / 411, G(2000, 0.25) 1311 / 1230 / 916, K(1000, 1000)
//   1593 / 2630 / 3413, 500 hubs joined to 2000 1262 / 2232 / 1322; where the
//   matrices are small, K(200, 800) 276 / 359 / 262, K(250, 1500) 609 / 915 / 574,
//   K(200, 1500) 438 / 765 / 529, 150 hubs joined to 1500 394 / 527 / 438.
//   Unions fill the GPU with units too small for the passes' CTAs: 2000 graphs
//   G(1100, 0.011), 29.6 ms with passes, 15.0 with rows.
inline SmallRoute small_route(int32_t n, int32_t G, int64_t n2, int64_t m, int32_t kmax, double d2, double kd) {
  if (n > kSmemTableMax || kmax < 2) return kRoutePasses;
  const double edges2 = 2.0 * (double)m;
  if (G > 1) return kRouteRows;
  if (n >= 64 && n <= kDenseMaxN && kmax <= kDenseMaxK && edges2 >= 0.15 * (double)n2 &&
      (d2 <= 8.0 * kd || (kmax <= 256 && edges2 >= 0.22 * (double)n2)))
    return kRouteDense;
  if (d2 <= 3.3e8 && kd <= 3e7) return kRouteRows;
  return d2 <= 7.0 * kd && edges2 >= 0.2 * (double)n2 ? kRouteRows : kRoutePasses;
}

// ---- host helpers (gc_api.cu) ----
void set_error(const std::string& msg);
// What a C entry answers to a C++ exception: GC_ERR_NOMEM, with a message if there is memory for one.
gc_status no_memory() noexcept;
gc_status cuda_fail(cudaError_t e, const char* what);

// The library's stream-ordered memory pool on the current device (created on
// first use). Freed blocks stay in it, up to a limit (environment
// GC_POOL_KEEP_BYTES; default a quarter of the device's memory), so that a
// later graph or count reuses them without mapping memory again and a free
// does not unmap at the next synchronisation; gc_release_cached_memory hands
// them back. Every device buffer of the library comes from it (pool_alloc),
// and is returned with cudaFreeAsync.
cudaMemPool_t lib_pool();
template <class T>
inline cudaError_t pool_alloc(T** p, size_t bytes, cudaStream_t s) {
  cudaMemPool_t pool = lib_pool();
  if (!pool) return cudaErrorMemoryAllocation;
  return cudaMallocFromPoolAsync(reinterpret_cast<void**>(p), bytes, pool, s);
}

// ---- host threads (gc_host.cu) ----
int host_threads();  // the cores of the host, at most 32
// f(0) .. f(n - 1) on the library's host threads and the calling thread; the
// calls of one host_run start in order. The first exception is thrown again
// here, after all have ended. Any thread may call it.
void host_run(int n, const std::function<void(int)>& f);

// ---- relabelling P1: the host half (gc_api.cu) ----
// Host arrays left uninitialised on allocation (every element is written
// before use).
template <class T>
struct HostBuf {
  std::unique_ptr<T[]> p;
  T* data() { return p.get(); }
  T& operator[](size_t i) { return p[i]; }
  void resize(size_t n) { p.reset(new T[n > 0 ? n : 1]); }
};
// Vertices ranked by ascending (degree, id) -- a stable counting sort of the
// degrees -- and what the device relabel needs: internal row pointers, and the
// internal rows of more than 32 entries listed by the sort that takes them.
struct RelabelPlan {
  HostBuf<int32_t> perm, newid, rp;
  std::vector<int32_t> mid, longr;  // rows of 33..4096 entries, and longer ones
  std::vector<int64_t> long_off;    // offset of each long row's padded copy
  int64_t tmp_len = 0;
  int32_t obound[kOBounds] = {};    // first rank of degree >= kOBoundDeg[k]
};
// On at most max_threads host threads. Throws std::bad_alloc.
RelabelPlan plan_relabel(int32_t n, const int32_t* rp, int max_threads);

// ---- relabelling P1 on the device (gc_relabel.cu) ----
// Internal row i = caller row perm[i] in internal ids (newid), sorted; eid:
// caller's edge id of every internal slot, or nullptr (not wanted). A union of
// graphs (vgid, gbase: of the internal ids) has caller columns local to their
// graph, and every other id global. rp: internal row pointers (device);
// mid_rows / long_rows: internal rows of 33..4096 and of more entries; the
// long rows are sorted in padded copies at tmp + long_off[k].
gc_status relabel_on_device(int32_t n, int32_t m, const int32_t* d_rp0, const int32_t* d_ci0,
                            const int32_t* d_perm, const int32_t* d_newid, const int32_t* d_rp, int32_t* d_ci,
                            int32_t* d_eid, const int32_t* d_vgid, const int32_t* d_gbase, const int32_t* d_mid_rows, int32_t n_mid, const int32_t* d_long_rows,
                            const int64_t* d_long_off, int32_t n_long, long long* d_tmp, cudaStream_t s);

// ---- preprocessing (gc_prep.cu) ----
struct PrepBuffers {
  int32_t* deg = nullptr;
  int32_t* eid = nullptr;
  int32_t* uv = nullptr;  // [m][2]
  int32_t* out_ptr = nullptr;
  int32_t* out_idx = nullptr;
  int32_t* units = nullptr;
  int32_t n_units = 0;
  int32_t dmax = 0;
  int32_t* rev = nullptr;  // [2m] slot of the reverse direction of every slot
  int32_t* ocsr = nullptr;  // [m] out-slot -> CSR slot
  int32_t* e2o = nullptr;   // [m] edge id -> out-slot
  int32_t* kunits = nullptr;  // pass K units (see CountArgs::kunits)
  int32_t ktier_off[kNumTiers + 1] = {0, 0, 0, 0, 0, 0};
  int32_t kmax = 0;         // largest out-degree
  int32_t* cunits = nullptr;  // pass C units: hub units (heaviest first), hashed units (heaviest
                              // first), then the rest in unit order
  int32_t n_cheavy = 0;
  int4* cjobs = nullptr;       // hub jobs, heaviest first (see CountArgs)
  int32_t n_cjobs = 0;
  int32_t* chash_w = nullptr;  // wedges of each hashed unit (both hash tiers)
  int32_t n_chash = 0;
  int32_t n_chash_mid = 0;     // hashed units of more than kHashMidW wedges
  int32_t n_chash_big = 0;     // hashed units of more than kHashSmallW wedges
  int32_t n_chash2 = 0;        // units of the packed-key hash tier
  int32_t n_chash2_big = 0;    // of them, units of more than kHash2HalfMaxW wedges
  int32_t n_cunits = 0;
  SmallRoute route = kRoutePasses;  // how the graph is counted (small_route)
  uint32_t* bits = nullptr;    // kRouteDense: bit rows, and the same by word (see DevGraph)
  uint32_t* bits_t = nullptr;
  HubGeom* hgeom = nullptr;    // layout of the hub kernel's o-range (owns hseg's block)
  HubSeg* hseg = nullptr;
  int32_t* hpos = nullptr;
};
// What the host knows of a ranked graph (ids = ranks, rows ascending) when it
// is prepared.
struct RankInfo {
  const int32_t* rp;      // [n + 1] internal row pointers
  int32_t G;              // graphs, each a range of ids
  const int32_t* gbase;   // [G] first id of each, ascending
  const int32_t* gn;      // [G] vertices of each
  const int32_t* obound;  // [G][kOBounds] first id of degree >= kOBoundDeg[k] (the graph's end if none)
  const int32_t* d_vgid;  // on the device: graph of every vertex, and gbase; nullptr for one graph
  const int32_t* d_gbase;
};
// Whether some pass-C units are left for the vertex-indexed tables.
inline bool needs_tables(const PrepBuffers& p) { return p.n_cunits > p.n_cheavy + p.n_chash + p.n_chash2; }
// Builds degrees, the degree-oriented out-lists, the reverse-slot map and the
// binned unit lists of a ranked graph on `stream`. d_eid (optional): slot ->
// edge id from the relabel (ownership passes to PrepBuffers); with it, and
// d_perm (internal -> caller vertex id), the edge list in the caller's labels
// and the edge id -> out-slot map are made too.
gc_status prepare_graph(int32_t n, int32_t m, const int32_t* d_rp, const int32_t* d_ci, int32_t* d_eid,
                        const int32_t* d_perm, const RankInfo& rank, PrepBuffers* out, cudaStream_t stream);
// Splits the pass-C units of a ranked graph (ids = ranks, rows ascending)
// into hub units for the blocked kernel, units of at most kHashMaxW wedges
// for the hashed kernel and the rest, leaving out units without wedges
// (fills cunits, n_cheavy, chash_w, n_chash, n_cunits; otherwise
// cunits is a copy of units).
gc_status classify_c_units(int32_t n, const int32_t* d_rp, const int32_t* d_ci, const RankInfo& rank, PrepBuffers* p,
                           cudaStream_t stream);
void free_prep(PrepBuffers* p, cudaStream_t s);
// Smallest slot p with rev[p] == p (no reverse: the input is not symmetric),
// or -1 (synchronises the stream).
gc_status first_unreversed_slot(int64_t nnz, const int32_t* d_rev, int32_t* out, cudaStream_t s);

// ---- small graphs on a shared-memory bitmatrix (gc_small.cu) ----
// Size classes of the bitmatrix kernel: class c takes graphs of at most
// kSmallClassN[c] vertices (and more than the previous class).
constexpr int kSmallClasses = 5;
constexpr int kSmallClassN[kSmallClasses] = {64, 128, 256, 512, 1024};
// Tunable parameters of the batched form (read from the tuning cache at
// gc_batch_create, or set with gc_batch_set_param).
struct BatchConfig {
  int32_t small_n_max = 512;                                  // graphs up to this many vertices: bitmatrix kernels
  int32_t class_block[kSmallClasses] = {256, 256, 256, 256, 256};  // threads per CTA of each size class
  int32_t use_graph = 1;                                      // replay each small-graph launch as a CUDA graph
  int32_t max_inflight = 2;                                   // launches the dispatcher keeps in flight
};
constexpr int kMaxInflight = 4;                                 // stream slots of a batch runtime
// Size class of a graph with n vertices (kSmallClasses if above the largest).
int small_class_of(int32_t n);
// Overrides cfg with the tuning cache's entry for the current GPU (gc_tune.cu);
// false (cfg unchanged) when there is no cache or no entry.
bool load_tuned_config(BatchConfig* cfg, std::string* source);
// Raises the dynamic shared-memory limit of every instantiation (once per
// device, before any launch or capture).
gc_status small_graphs_setup();
// The units of a launch of small graphs (n, m per graph): unit = (graph, part |
// parts << 16), class c's units[class_off[c] .. class_off[c + 1]), most work
// first within a class.
void small_units(const std::vector<int32_t>& n, const std::vector<int64_t>& m, std::vector<int2>* units,
                 int32_t* class_off);
constexpr int kSmallSums = 8;  // sums of a graph that the kernels leave in SmallGraphs::sums
// Device arrays of one launch: rp/voff: concatenated local row pointers and
// their offsets; ci/eoff: concatenated local columns; gn/gm: vertices and edges
// per graph; cursor: kSmallClasses zeroed ints; status: device status word;
// sums [G][kSmallSums] zeroed; csum [G][13][2] receives the unrestricted sums.
struct SmallGraphs {
  int32_t G;
  const int32_t *rp, *ci, *gn;
  const int64_t *voff, *eoff, *gm;
  const int2* units;
  int32_t *cursor, *status;
  unsigned long long *sums, *csum;
};
// Streams on which the size classes of one launch run side by side.
struct SmallFork {
  cudaEvent_t start = nullptr, done[kSmallClasses] = {};
  cudaStream_t stream[kSmallClasses] = {};
};
// ev (optional): 2 kSmallClasses events, recorded before and after each class's
// kernel; fork (optional): the classes run on its streams, joined into s.
gc_status run_small_graphs(const SmallGraphs& b, const int32_t* class_off, const BatchConfig& cfg, cudaEvent_t* ev,
                           const SmallFork* fork, cudaStream_t s);

// ---- counting (gc_count.cu: pass C, finish, derive; gc_clique.cu: passes T and K) ----
int count_grid_size();
gc_status run_pass_c(const DevGraph& g, const CountArgs& a, cudaStream_t s);
gc_status run_pass_c_heavy(const DevGraph& g, const CountArgs& a, cudaStream_t s);
// |T|, the 4-cycles and the cross terms of every edge, for unions of graphs of
// at most kSmemTableMax vertices; and the 4-cliques without pass T.
gc_status run_rows(const DevGraph& g, const CountArgs& a, cudaStream_t s);
gc_status run_cliques_alone(const DevGraph& g, const CountArgs& a, Fork* fork, int* launches);
// The same two for a dense graph, on its bit rows: k_rows_dense reads them
// instead of the neighbours' lists, k_cliques_dense packs every H_a from them.
gc_status run_rows_dense(const DevGraph& g, const CountArgs& a, cudaStream_t s);
gc_status run_cliques_dense(const DevGraph& g, const CountArgs& a, int32_t kmax, cudaStream_t s);
// Bit rows of a prepared graph of at most kDenseMaxN vertices (P->bits, bits_t).
gc_status build_bits(int32_t n, const int32_t* d_rp, const int32_t* d_ci, PrepBuffers* p, cudaStream_t s);
constexpr int kHeavyTab = 53248;  // largest o-range block of the hub kernel of pass C (words of shared memory)
// Words of the hub kernel's count block (environment GC_HUB_TAB_WORDS, a
// multiple of 1024 in [4096, kHeavyTab], else kHubTabDefault), read once per
// process. The block and the SM's L1 cache share one array, split in steps
// (the shared-memory carveout); kHubTabDefault with the kernel's 8.2 KB of
// static arrays and 1 KB reserved fits the 196 KB step, leaving about 60 KB of
// L1 for the rows instead of 28 KB with a 208 KB block (R-MAT scale 22, when
// blocks had one counter width: pass C 228.4 ms at 53248 words, 205.0 at 45056,
// 213.3 at 39936, 226.7 at 32768; now 139 at 45056 and at 47104, the largest
// that fits).
constexpr int kHubTabDefault = 45056;
int hub_tab_words();
// Counters per word that a unit of nx lower neighbours could use over its
// whole o-range by nx alone; the rule that picks the hub units estimates
// their blocks with it. It dates from blocks of one counter width: with segments
// there are fewer blocks (8 where it says 31 to 94 on R-MAT scale 22), and the
// line between the hub kernel and the others was not measured again.
__host__ __device__ __forceinline__ int hub_cpw(int64_t nx) { return nx < 1023 ? 3 : nx < 65536 ? 2 : 1; }
// Units of pass C with at most kHashMaxW wedges count in a shared-memory
// hash of 2 kHashMaxW keys (at most half full: a unit has no more distinct
// o than wedges).
constexpr int kHashMaxW = 8192;
constexpr int kHashSmallW = 512;  // hashed units up to this many wedges run in small CTAs
constexpr int kHashMidW = 2048;   // and up to this many in middle-sized CTAs
gc_status run_pass_c_hash(const DevGraph& g, const CountArgs& a, Fork* fork, int* launches);
// Units of more than kHashMaxW and at most kHash2MaxW wedges, with fewer than
// kHash2MaxNx lower neighbours, in graphs of at most 2^22 vertices: a
// shared-memory hash of kHash2Slots words, each a packed (22-bit vertex,
// 10-bit count) pair, at most 72 % full.
constexpr int kHash2Slots = 57344;
constexpr int kHash2MaxW = 41287;
constexpr int kHash2MaxNx = 1023;
// Packed-key units of at most kHash2HalfMaxW wedges fit half the table and
// run in 512-thread CTAs, two an SM.
constexpr int kHash2HalfSlots = 28672;
constexpr int kHash2HalfMaxW = 20620;  // (kHash2HalfSlots - 32) * 18 / 25
constexpr int32_t kHash2MaxN = 1 << 22;
gc_status run_pass_c_hash2(const DevGraph& g, const CountArgs& a, Fork* fork, int* launches);
gc_status run_derive(const DevGraph& g, const unsigned long long* csum, unsigned long long* x,
                     int32_t* status, cudaStream_t s);
// The tiers of passes T and K: side by side on the fork's streams.
gc_status run_pass_t(const DevGraph& g, const CountArgs& a, Fork* fork, int* launches);
gc_status run_pass_k(const DevGraph& g, const CountArgs& a, Fork* fork, int* launches);
gc_status run_finish(const DevGraph& g, const CountArgs& a, cudaStream_t s);
// Per-edge induced counts of H_7..H_16 (needs a.dsum from pass T, and the
// results of passes C and K); vsum: [n][2] scratch.
gc_status run_induced(const DevGraph& g, const CountArgs& a, unsigned long long* vsum, uint64_t* out, bool out_host,
                      cudaStream_t s);
// Bytes of one global-tier buffer for out-degrees up to cap.
size_t kbuf_bytes(int32_t cap);
// Ordering key of the units on the vertex-indexed tables (environment GC_ORDER):
// 0 = vol (default: d_v^2, heaviest bin first), 1 = degree d_v, 2 = none (vertex id).
int order_key();
// exclusive prefix sum of n int32 into out[0..n] (out[n] = total)
gc_status exclusive_scan(int32_t n, const int32_t* in, int32_t* out, cudaStream_t s);

}  // namespace gc
