// gc_batch.cu -- batched and served counting of many graphs (see include/gc.h).
//
// A launch counts all graphs taken from the pending queue as one disjoint
// union: graph g keeps its vertices in the global range [gbase[g],
// gbase[g] + n_g). Triangles, 4-cliques and 4-cycles of a disjoint union are
// those of its components, so the per-edge kernels run unchanged over the
// union -- one persistent grid per pass, CTAs stealing v-groups of every graph
// from one difficulty-binned queue -- while the per-edge columns use each
// graph's own n and m and the unrestricted counts are summed per graph.
//
// Continuous batching: submit() admits a graph while the admitted graphs'
// estimated device footprint stays within the budget; a dispatcher thread
// launches whatever is pending whenever fewer than two launches are in
// flight (each launch on its own stream, so a new launch's preparation
// overlaps the previous launch's counting) and retires finished launches,
// which releases their share of the budget.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <iterator>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <unordered_map>
#include <vector>

#include "gc_deal.h"
#include "gc_internal.h"

namespace gc {
gc_status validate_csr(int32_t n, const int32_t* rp, const int32_t* ci);
gc_status validate_csr_small(int32_t n, const int32_t* rp, const int32_t* ci, std::vector<int32_t>* fill);

namespace {

// The checks of one graph on the device, thread per slot: *bad becomes non-zero
// if a column is out of range, a self-loop, not above its predecessor, or its
// reverse is absent (row pointers from 0 to nnz, ascending, are checked
// before). The host's walk over the reverses waits on memory once per edge:
// 6.2 ms for 3.5M entries on 16 cores, against 0.9 ms for copy and kernel.
__global__ void __launch_bounds__(256) k_check_csr(int32_t n, int32_t nnz, const int32_t* __restrict__ rp,
                                                   const int32_t* __restrict__ ci, int32_t* __restrict__ bad) {
  const int lane = threadIdx.x & 31;
  bool ok = true;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p - lane < nnz; p += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p0 = (int32_t)(p - lane), p_last = (int32_t)min((int64_t)p0 + 31, (int64_t)nnz - 1);
    const int32_t q = (int32_t)min(p, (int64_t)nnz - 1);
    const int32_t x = row_of_slot(n, rp, p0, q, p_last);
    const int32_t y = ci[q];
    if ((uint32_t)y >= (uint32_t)n || y == x || (q > rp[x] && ci[q - 1] >= y)) {
      ok = false;
      continue;
    }
    int32_t lo = rp[y];
    const int32_t ye = rp[y + 1];
    for (int32_t hi = ye; lo < hi;) {
      const int32_t mid = lo + ((hi - lo) >> 1);
      if (ci[mid] < x) lo = mid + 1; else hi = mid;
    }
    ok &= lo < ye && ci[lo] == x;
  }
  if (!ok) *bad = 1;
}

// A batch may be used while some thread captures a stream of its own: its work is
// on other streams, so that its allocations, queries and waits may run then, which
// the runtime wants to be told (else it refuses them and ends the capture, also
// when it is another thread's in the default, global mode). Held by every call
// that does such things and by the dispatcher all its life.
struct OutsideCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~OutsideCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// The library's host copy of one submission, pinned where possible, so that a
// launch copies it to the device directly.
struct HostBlock {
  int32_t* p = nullptr;
  size_t cap = 0;
  bool pinned = false;
};

void free_block(const HostBlock& h) {
  if (h.pinned) {
    OutsideCapture relaxed;
    cudaFreeHost(h.p);
  } else {
    delete[] h.p;
  }
}

// Host blocks of retired submissions, kept for reuse: a submission takes the
// smallest kept block that holds it and is not more than twice as large, whose
// pages are already mapped and pinned, instead of a fresh allocation. Blocks are
// not initialised (the copy that fills one writes every entry it reads). A
// returned block is kept whatever the number, since giving pinned memory back
// waits for the whole device; trim(), called without any lock when the batch has
// nothing to do, keeps at most kLarge blocks of kLargeEntries or more and kSmall
// others, the largest. The cache lives until the batch and its last block are gone.
struct HostCache {
  static constexpr size_t kLarge = 4, kSmall = 64;
  static constexpr size_t kLargeEntries = (size_t)16 << 20;
  std::mutex mu;
  std::multimap<size_t, HostBlock> free;  // by capacity
  ~HostCache() {
    for (auto& h : free) free_block(h.second);
  }
  void put(const HostBlock& h) {
    try {
      std::lock_guard<std::mutex> lk(mu);
      free.emplace(h.cap, h);
      return;
    } catch (...) {  // no memory to keep it
    }
    free_block(h);
  }
  void trim() {
    for (;;) {
      HostBlock out;
      {
        std::lock_guard<std::mutex> lk(mu);
        const auto large = free.lower_bound(kLargeEntries);
        const size_t n_large = (size_t)std::distance(large, free.end());
        auto it = n_large > kLarge ? large : free.size() - n_large > kSmall ? free.begin() : free.end();
        if (it == free.end()) return;
        out = it->second;
        free.erase(it);
      }
      free_block(out);
    }
  }
};

// A block of at least `entries` int32; it returns to the cache when its last
// reference goes. Throws std::bad_alloc.
std::shared_ptr<HostBlock> host_block(const std::shared_ptr<HostCache>& cache, size_t entries) {
  if (entries == 0) entries = 1;
  if (entries < 4096) {  // not worth pinning
    HostBlock h;
    h.p = new int32_t[entries];
    h.cap = entries;
    return std::shared_ptr<HostBlock>(new HostBlock(h), [](HostBlock* q) {
      free_block(*q);
      delete q;
    });
  }
  HostBlock h;
  {
    std::lock_guard<std::mutex> lk(cache->mu);
    const auto it = cache->free.lower_bound(entries);
    if (it != cache->free.end() && it->first / 2 <= entries) {
      h = it->second;
      cache->free.erase(it);
    }
  }
  if (!h.p) {
    h.cap = entries + entries / 8;
    OutsideCapture relaxed;
    if (cudaHostAlloc(reinterpret_cast<void**>(&h.p), sizeof(int32_t) * h.cap, cudaHostAllocPortable) == cudaSuccess) {
      h.pinned = true;
    } else {
      cudaGetLastError();
      h.p = new int32_t[h.cap];
    }
  }
  std::shared_ptr<HostCache> keep = cache;
  return std::shared_ptr<HostBlock>(new HostBlock(h), [keep](HostBlock* q) {
    const HostBlock out = *q;
    delete q;
    keep->put(out);
  });
}

// A graph waiting for a launch. Its CSR is the library's own copy: rp (n + 1
// entries starting at 0) and ci (2m entries) point into `owner` -- a copy of
// one graph (gc_batch_submit), or one shared copy of a whole bulk submission
// (gc_batch_submit_many: all row pointers, then all columns, copied while
// validating).
struct PendingGraph {
  uint64_t ticket;
  int32_t n;
  int64_t m;
  int64_t bytes;
  const int32_t* rp = nullptr;
  const int32_t* ci = nullptr;
  std::shared_ptr<HostBlock> owner;
};

// Results of one launch ([G][17][2]), shared by its tickets until they retire.
typedef std::vector<uint64_t> Results;

struct Ticket {
  enum State : uint8_t { kRetired = 0, kLive, kDone };
  State state = kRetired;
  gc_status status = GC_OK;
  int32_t slot = 0;  // row in *out
  std::shared_ptr<Results> out;
};

// One check of a submission on the device (checked_on_device).
struct Check {
  cudaStream_t stream = nullptr;     // of high priority, so that it does not wait behind the launches in flight
  cudaEvent_t done = nullptr;
  int32_t* bad = nullptr;            // pinned
  int32_t* d = nullptr;              // flag, row pointers, columns
  std::shared_ptr<HostBlock> own;    // what the device reads, until the check is over
  bool busy = false;
};
// Checks at a time; a submission that finds them all busy is checked on the host.
constexpr int kChecks = 4;

// Timers of one launch (CUDA events on its stream): the size classes of the
// small-graph kernels (eager launches only), the whole small-graph sequence
// (copies in, kernels, derive, copy out) and the larger graphs' passes.
enum { kEvSmall0 = 0, kEvSmallSeq0 = 2 * kSmallClasses, kEvSmallSeq1, kEvUnion0, kEvUnion1, kNumLaunchEv };

struct Launch {
  std::vector<uint64_t> tickets;
  std::vector<int32_t> slot;          // ticket k's row in h_x
  int64_t bytes = 0;
  int stream_slot = 0;
  BatchConfig cfg;                    // the batch's parameters when the launch was taken
  cudaStream_t stream = nullptr;
  cudaEvent_t done = nullptr;
  cudaEvent_t ev[kNumLaunchEv] = {};
  bool timed_classes = false, timed_small = false, timed_union = false, replayed = false;
  unsigned long long* h_x = nullptr;  // pinned [G][17][2], cap_x graphs
  size_t cap_x = 0;
  int32_t* h_status = nullptr;        // pinned: small graphs, union
  std::vector<std::shared_ptr<HostBlock>> owners;  // the device copies from them until the launch is done
  gc_status launch_status = GC_OK;
  std::string error;
};

// Device buffers and pinned host staging of the small-graph path, one set per
// stream slot, grown as needed and kept: once warm, a launch allocates
// nothing, and its sequence (copies in, kernels, derive, copy out) can be
// captured and replayed as a CUDA graph. `busy` marks the end of the slot's
// last sequence: the host waits on it before it refills or regrows them.
struct SmallBufs {
  size_t cap_rows = 0, cap_nnz = 0, cap_hrows = 0, cap_hnnz = 0, cap_g = 0, cap_units = 0;
  int32_t *d_rp = nullptr, *d_ci = nullptr, *d_gn = nullptr, *d_misc = nullptr;
  int2 *d_units = nullptr, *h_units = nullptr;
  int64_t *d_voff = nullptr, *d_eoff = nullptr, *d_gm = nullptr;
  unsigned long long *d_sums = nullptr, *d_csum = nullptr, *d_x = nullptr;
  int32_t *h_rp = nullptr, *h_ci = nullptr, *h_gn = nullptr;
  int64_t *h_voff = nullptr, *h_eoff = nullptr, *h_gm = nullptr;
  cudaGraphExec_t exec = nullptr;
  cudaEvent_t busy = nullptr;
  SmallFork fork;
};

void free_small_bufs(SmallBufs* b) {
  if (b->busy) cudaEventSynchronize(b->busy);
  for (void* p : {(void*)b->d_rp, (void*)b->d_ci, (void*)b->d_units, (void*)b->d_gn, (void*)b->d_misc,
                  (void*)b->d_voff, (void*)b->d_eoff, (void*)b->d_gm, (void*)b->d_sums, (void*)b->d_csum,
                  (void*)b->d_x})
    if (p) cudaFree(p);
  for (void* p : {(void*)b->h_rp, (void*)b->h_ci, (void*)b->h_units, (void*)b->h_gn, (void*)b->h_voff,
                  (void*)b->h_eoff, (void*)b->h_gm})
    if (p) cudaFreeHost(p);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->busy) cudaEventDestroy(b->busy);
  if (b->fork.start) cudaEventDestroy(b->fork.start);
  for (auto& e : b->fork.done)
    if (e) cudaEventDestroy(e);
  for (auto& t : b->fork.stream)
    if (t) cudaStreamDestroy(t);
  *b = SmallBufs();
}

int64_t footprint(int32_t n, int64_t m) {
  int64_t b = 44LL * n + 32LL * m + 1024;
  if (n > kSmemTableMax) b += (int64_t)count_grid_size() * n * 4;
  return b;
}

}  // namespace
}  // namespace gc

using namespace gc;

struct gc_batch_s {
  int64_t budget = 0;
  uint32_t flags = 0;
  BatchConfig cfg;
  SmallBufs small[kMaxInflight];        // per stream slot
  ForkSet* forks[kMaxInflight] = {};    // per stream slot, of the larger graphs' launches
  double last_stats[GC_BATCH_STATS] = {};  // of the last retired launch
  int64_t in_use = 0;
  std::mutex mu;
  std::condition_variable cv;
  // the budget: admitted graphs, and submissions still being checked
  bool reserve(int64_t bytes) {
    std::lock_guard<std::mutex> lk(mu);
    if (in_use + bytes > budget) return false;
    in_use += bytes;
    return true;
  }
  void release(int64_t bytes) {
    {
      std::lock_guard<std::mutex> lk(mu);
      in_use -= bytes;
    }
    cv.notify_all();
  }
  std::deque<PendingGraph> pending;
  std::vector<Launch*> inflight;
  std::deque<Ticket> tickets;           // of the numbers first_ticket .. (the oldest one unretired or later)
  uint64_t first_ticket = 1;
  size_t live = 0;                      // tickets not retired
  std::unordered_map<uint64_t, Ticket> old;  // unretired tickets below first_ticket, long unpolled
  std::vector<Launch*> spare;           // retired launches, for their events and pinned results (trimmed to kMaxSpare)
  Ticket* find(uint64_t t) {            // nullptr: unknown or retired
    if (t < first_ticket) {
      const auto it = old.find(t);
      return it == old.end() ? nullptr : &it->second;
    }
    if (t - first_ticket >= tickets.size()) return nullptr;
    Ticket* k = &tickets[(size_t)(t - first_ticket)];
    return k->state == Ticket::kRetired ? nullptr : k;
  }
  uint64_t add_ticket() {
    tickets.emplace_back();
    tickets.back().state = Ticket::kLive;
    ++live;
    return first_ticket + tickets.size() - 1;
  }
  // A place at the end of the queue, and its ticket; or neither, and an exception.
  uint64_t admit() {
    pending.emplace_back();
    try {
      return add_ticket();
    } catch (...) {
      pending.pop_back();
      throw;
    }
  }
  void dismiss() {  // the last admitted
    pending.pop_back();
    tickets.pop_back();
    --live;
  }
  void retire(uint64_t t) {
    if (t < first_ticket) old.erase(t);
    else tickets[(size_t)(t - first_ticket)] = Ticket();
    --live;
  }
  // A ticket that is never polled does not keep all later ones: where most of the
  // queue is retired, its oldest move out of it.
  void drop_retired() {
    while (!tickets.empty()) {
      Ticket& f = tickets.front();
      if (f.state != Ticket::kRetired) {
        if (tickets.size() <= 4096 + 2 * live) break;
        try {
          old.reserve(old.size() + 1);  // nothing is moved before all memory is there
          old.emplace(first_ticket, std::move(f));
        } catch (...) {
          break;  // no memory for it: it stays
        }
      }
      tickets.pop_front();
      ++first_ticket;
    }
  }
  bool stop = false;
  std::thread dispatcher;
  std::mutex check_mu;                  // of the checks' busy marks
  Check checks[kChecks];
  cudaStream_t streams[kMaxInflight] = {};
  int next_stream = 0;                  // manual mode: round-robin over the slots
  int device = 0;
  std::shared_ptr<HostCache> host = std::make_shared<HostCache>();  // submissions' copies
};
static constexpr size_t kMaxSpare = 8;

namespace {

// Counts `graphs` as one launch on `s`. Fills L (results land in L->h_x when
// L->done completes). Runs in the dispatcher thread (or the flushing thread
// in manual mode) without holding the batch lock.
// The graphs too large for the bitmatrix kernel, as one disjoint union
// through the general passes. Results go to h_x_dst ([G][17][2], pinned) and
// the launch status word to *h_status_dst.
gc_status run_union(std::vector<PendingGraph*>& graphs, cudaStream_t s, ForkSet* fs, Launch* L,
                    unsigned long long* h_x_dst, int32_t* h_status_dst) {
  const int32_t G = (int32_t)graphs.size();
  int64_t n_total = 0, nnz_total = 0;
  int32_t table_n = 0;
  for (auto* pg : graphs) {
    n_total += pg->n;
    nnz_total += 2 * pg->m;
    if (pg->n > table_n) table_n = pg->n;
  }
  const int32_t n = (int32_t)n_total;
  const int32_t m = (int32_t)(nnz_total / 2);
  // The union is ranked like a single graph (P1), graph by graph: the ids of
  // graph g are gbase[g] + the (degree, id) rank in g, so that the hub and hash
  // kernels of pass C serve it too. (Unranked, with pass C on vertex-indexed
  // tables in DRAM, 40 Chung-Lu graphs of 1 000 to 2M edges took 29 ms in pass C
  // alone.) Host arrays, one block: gbase | gn | obound, then per vertex.
  std::vector<int32_t> gbase((size_t)G + 1), gn((size_t)G), obound((size_t)G * kOBounds);
  std::vector<int64_t> gm((size_t)G), ebase((size_t)G + 1);
  gbase[0] = 0;
  ebase[0] = 0;
  for (int32_t gi = 0; gi < G; ++gi) {
    gn[(size_t)gi] = graphs[(size_t)gi]->n;
    gm[(size_t)gi] = graphs[(size_t)gi]->m;
    gbase[(size_t)gi + 1] = gbase[(size_t)gi] + graphs[(size_t)gi]->n;
    ebase[(size_t)gi + 1] = ebase[(size_t)gi] + 2 * graphs[(size_t)gi]->m;
  }
  HostBuf<int32_t> h_rp, h_rp0, h_perm, h_newid, h_vgid;
  std::vector<int32_t> mid, longr;
  std::vector<int64_t> long_off;
  int64_t tmp_len = 0;
  try {
    for (auto* b : {&h_rp, &h_rp0, &h_perm, &h_newid, &h_vgid}) b->resize((size_t)n + 1);
    std::vector<RelabelPlan> plans((size_t)G);
    host_run(G, [&](int gi) {
      const PendingGraph& pg = *graphs[(size_t)gi];
      RelabelPlan& R = plans[(size_t)gi];
      R = plan_relabel(pg.n, pg.rp, 1);
      const int32_t vb = gbase[(size_t)gi], eb = (int32_t)ebase[(size_t)gi];
      for (int32_t i = 0; i < pg.n; ++i) {
        h_rp[(size_t)(vb + i)] = eb + R.rp[(size_t)i];
        h_rp0[(size_t)(vb + i)] = eb + pg.rp[i];
        h_perm[(size_t)(vb + i)] = vb + R.perm[(size_t)i];
        h_newid[(size_t)(vb + i)] = vb + R.newid[(size_t)i];
        h_vgid[(size_t)(vb + i)] = gi;
      }
      for (int k = 0; k < kOBounds; ++k) obound[(size_t)gi * kOBounds + (size_t)k] = vb + R.obound[k];
    });
    h_rp[(size_t)n] = h_rp0[(size_t)n] = (int32_t)nnz_total;
    for (int32_t gi = 0; gi < G; ++gi) {
      const RelabelPlan& R = plans[(size_t)gi];
      for (int32_t x : R.mid) mid.push_back(gbase[(size_t)gi] + x);
      for (int32_t x : R.longr) longr.push_back(gbase[(size_t)gi] + x);
      for (int64_t o : R.long_off) long_off.push_back(tmp_len + o);
      tmp_len += R.tmp_len;
    }
  } catch (...) {
    set_error("host allocation failed");
    L->error = gc_last_error();
    return GC_ERR_NOMEM;
  }
  const size_t n1 = (size_t)n + 1, nnz1 = (size_t)(nnz_total > 0 ? nnz_total : 1);
  const size_t n_lists = mid.size() + longr.size();
  int32_t *d_rp = nullptr, *d_ci = nullptr, *d_vgid = nullptr, *d_desc = nullptr, *d_rp0 = nullptr, *d_ci0 = nullptr;
  int32_t *d_perm = nullptr, *d_newid = nullptr, *d_lists = nullptr;
  int64_t *d_gm = nullptr, *d_loff = nullptr;
  long long* d_tmp = nullptr;
  RankInfo rank = RankInfo();
  PrepBuffers prep;
  Scratch sc;
  cudaError_t e = cudaSuccess;
  gc_status st = GC_OK;
  auto fail = [&](cudaError_t err, const char* what) {
    st = cuda_fail(err, what);
    L->error = gc_last_error();
  };
  auto up = [&](auto* d, const auto* h, size_t count) {
    return count ? cudaMemcpyAsync(d, h, sizeof(*h) * count, cudaMemcpyHostToDevice, s) : cudaSuccess;
  };
#define GB_TRY(call, what)  \
  do {                      \
    e = (call);             \
    if (e != cudaSuccess) { \
      fail(e, what);        \
      goto out;             \
    }                       \
  } while (0)
  GB_TRY(pool_alloc(&d_rp, sizeof(int32_t) * n1, s), "batch alloc");
  GB_TRY(pool_alloc(&d_ci, sizeof(int32_t) * nnz1, s), "batch alloc");
  GB_TRY(pool_alloc(&d_vgid, sizeof(int32_t) * n1, s), "batch alloc");
  GB_TRY(pool_alloc(&d_desc, sizeof(int32_t) * 2 * (size_t)G, s), "batch alloc");
  GB_TRY(pool_alloc(&d_gm, sizeof(int64_t) * (size_t)G, s), "batch alloc");
  GB_TRY(pool_alloc(&d_rp0, sizeof(int32_t) * n1, s), "batch alloc");
  GB_TRY(pool_alloc(&d_ci0, sizeof(int32_t) * nnz1, s), "batch alloc");
  GB_TRY(pool_alloc(&d_perm, sizeof(int32_t) * n1, s), "batch alloc");
  GB_TRY(pool_alloc(&d_newid, sizeof(int32_t) * n1, s), "batch alloc");
  GB_TRY(pool_alloc(&d_lists, sizeof(int32_t) * (n_lists + 1), s), "batch alloc");
  GB_TRY(pool_alloc(&d_loff, sizeof(int64_t) * (long_off.size() + 1), s), "batch alloc");
  GB_TRY(pool_alloc(&d_tmp, sizeof(long long) * (size_t)(tmp_len + 1), s), "batch alloc");
  for (int32_t gi = 0, gj; gi < G; gi = gj) {  // the columns, graphs that lie next to each other in one copy
    gj = gi + 1;
    while (gj < G && graphs[(size_t)gj]->ci == graphs[(size_t)gj - 1]->ci + 2 * gm[(size_t)gj - 1]) ++gj;
    GB_TRY(up(d_ci0 + ebase[(size_t)gi], graphs[(size_t)gi]->ci, (size_t)(ebase[(size_t)gj] - ebase[(size_t)gi])),
           "batch copy");
  }
  GB_TRY(up(d_rp, h_rp.data(), n1), "batch copy");
  GB_TRY(up(d_rp0, h_rp0.data(), n1), "batch copy");
  GB_TRY(up(d_perm, h_perm.data(), (size_t)n), "batch copy");
  GB_TRY(up(d_newid, h_newid.data(), (size_t)n), "batch copy");
  GB_TRY(up(d_vgid, h_vgid.data(), (size_t)n), "batch copy");
  GB_TRY(up(d_desc, gbase.data(), (size_t)G), "batch copy");
  GB_TRY(up(d_desc + G, gn.data(), (size_t)G), "batch copy");
  GB_TRY(up(d_gm, gm.data(), (size_t)G), "batch copy");
  GB_TRY(up(d_lists, mid.data(), mid.size()), "batch copy");
  GB_TRY(up(d_lists + mid.size(), longr.data(), longr.size()), "batch copy");
  GB_TRY(up(d_loff, long_off.data(), long_off.size()), "batch copy");
  rank = {h_rp.data(), G, gbase.data(), gn.data(), obound.data(), d_vgid, d_desc};
  if ((st = relabel_on_device(n, m, d_rp0, d_ci0, d_perm, d_newid, d_rp, d_ci, nullptr, d_vgid, d_desc, d_lists,
                              (int32_t)mid.size(), d_lists + mid.size(), d_loff, (int32_t)longr.size(), d_tmp, s)) !=
          GC_OK ||
      (st = prepare_graph(n, m, d_rp, d_ci, nullptr, nullptr, rank, &prep, s)) != GC_OK) {
    L->error = gc_last_error();
    goto out;
  }
  for (void* p : {(void*)d_rp0, (void*)d_ci0, (void*)d_perm, (void*)d_newid, (void*)d_lists, (void*)d_loff, (void*)d_tmp})
    cudaFreeAsync(p, s);
  d_rp0 = d_ci0 = d_perm = d_newid = d_lists = nullptr;
  d_loff = nullptr;
  d_tmp = nullptr;
  if ((st = scratch_init(&sc, m, needs_tables(prep) ? table_n : 0, prep.kmax, prep.ktier_off, G, 0, s)) != GC_OK) {
    L->error = gc_last_error();
    goto out;
  }
  {
    DevGraph dg;
    dg.n = n;
    dg.m = m;
    dg.rp = d_rp;
    dg.ci = d_ci;
    dg.deg = prep.deg;
    dg.eid = prep.eid;
    dg.out_ptr = prep.out_ptr;
    dg.out_idx = prep.out_idx;
    dg.ocsr = prep.ocsr;
    dg.e2o = prep.e2o;
    dg.rev = prep.rev;
    dg.G = G;
    dg.vgid = d_vgid;
    dg.gbase = d_desc;
    dg.gn = d_desc + G;
    dg.gm = d_gm;
    dg.table_n = table_n;
    dg.bits = dg.bits_t = nullptr;
    dg.hgeom = prep.hgeom;
    dg.hseg = prep.hseg;
    dg.hpos = prep.hpos;
    dg.n_long = 0;  // for the induced counts, which unions do not have
    KUnits ku;
    ku.kmax = prep.kmax;
    ku.units = prep.kunits;
    ku.cunits = prep.cunits;
    ku.n_cheavy = prep.n_cheavy;
    ku.cjobs = prep.cjobs;
    ku.n_cjobs = prep.n_cjobs;
    ku.chash_w = prep.chash_w;
    ku.n_chash = prep.n_chash;
    ku.n_chash2 = prep.n_chash2;
    ku.n_chash_big = prep.n_chash_big;
    ku.n_chash_mid = prep.n_chash_mid;
    ku.n_chash2_big = prep.n_chash2_big;
    ku.n_cunits = prep.n_cunits;
    ku.rows = prep.route != kRoutePasses;
    for (int t = 0; t <= kNumTiers; ++t) ku.tier_off[t] = prep.ktier_off[t];
    if ((st = run_count(dg, prep.units, prep.n_units, ku, nullptr, &sc, s, fs, nullptr)) != GC_OK) {
      fork_drain(fs);
      L->error = gc_last_error();
      goto out;
    }
    GB_TRY(cudaMemcpyAsync(h_x_dst, sc.x, sizeof(unsigned long long) * (size_t)G * 34, cudaMemcpyDeviceToHost, s),
           "batch copy out");
    GB_TRY(cudaMemcpyAsync(h_status_dst, sc.misc + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, s), "batch copy out");
  }
out:
#undef GB_TRY
  free_prep(&prep, s);
  scratch_free(&sc, s);
  for (void* p : {(void*)d_rp, (void*)d_ci, (void*)d_vgid, (void*)d_desc, (void*)d_gm, (void*)d_rp0, (void*)d_ci0,
                  (void*)d_perm, (void*)d_newid, (void*)d_lists, (void*)d_loff, (void*)d_tmp})
    if (p) cudaFreeAsync(p, s);
  return st;
}

// Grows the device buffer *d and the pinned host buffer *h (either may be
// absent) to hold `need` elements of T.
template <typename T>
cudaError_t grow_pair(T** d, T** h, size_t* cap, size_t need) {
  if (need <= *cap && (d == nullptr || *d) && (h == nullptr || *h)) return cudaSuccess;
  const size_t want = need + need / 4 + 64;
  if (d && *d) cudaFree(*d);
  if (h && *h) cudaFreeHost(*h);
  if (d) *d = nullptr;
  if (h) *h = nullptr;
  *cap = 0;
  cudaError_t e = cudaSuccess;
  if (d) e = cudaMalloc(d, sizeof(T) * want);
  if (e == cudaSuccess && h) e = cudaMallocHost(h, sizeof(T) * want);
  if (e == cudaSuccess) *cap = want;
  return e;
}

// Graphs of at most cfg.small_n_max vertices: packed as they are (local ids)
// into the slot's pinned staging and counted one CTA per graph on a
// shared-memory bitmatrix, binned by size class. The sequence is captured
// into a CUDA graph and replayed (cudaGraphExecUpdate keeps one executable
// per slot while the shape of the launches stays the same), or issued
// eagerly with per-class timers when cfg.use_graph is 0.
gc_status run_small(std::vector<PendingGraph*>& graphs, cudaStream_t s, Launch* L, unsigned long long* h_x_dst,
                    SmallBufs* sb, const BatchConfig& cfg) {
  const int32_t G = (int32_t)graphs.size();
  std::vector<int64_t> voff((size_t)G + 1), eoff((size_t)G + 1);
  voff[0] = eoff[0] = 0;
  for (int32_t gi = 0; gi < G; ++gi) {
    voff[gi + 1] = voff[gi] + graphs[gi]->n + 1;
    eoff[gi + 1] = eoff[gi] + 2 * graphs[gi]->m;
  }
  const size_t rows = (size_t)voff[G], nnz = (size_t)(eoff[G] > 0 ? eoff[G] : 1);
  gc_status st = GC_OK;
  cudaError_t e = cudaSuccess;
#define GS_TRY(call, what)                   \
  do {                                       \
    e = (call);                              \
    if (e != cudaSuccess) {                  \
      st = cuda_fail(e, what);               \
      L->error = gc_last_error();            \
      return st;                             \
    }                                        \
  } while (0)
  // Graphs that lie one after another in one pinned block (a whole bulk
  // submission) are copied to the device from there; others are packed into
  // pinned staging first.
  bool direct = graphs[0]->owner && graphs[0]->owner->pinned;
  for (int32_t gi = 1; gi < G && direct; ++gi) {
    const PendingGraph &p = *graphs[(size_t)gi - 1], &q = *graphs[(size_t)gi];
    direct = q.owner == p.owner && q.rp == p.rp + p.n + 1 && q.ci == p.ci + 2 * p.m;
  }
  if (sb->busy) GS_TRY(cudaEventSynchronize(sb->busy), "small buffers in use");
  else GS_TRY(cudaEventCreateWithFlags(&sb->busy, cudaEventDisableTiming), "small event");
  {
    size_t cg = sb->cap_g;
    GS_TRY(grow_pair<int32_t>(&sb->d_rp, nullptr, &sb->cap_rows, rows), "small buffers");
    GS_TRY(grow_pair<int32_t>(&sb->d_ci, nullptr, &sb->cap_nnz, nnz), "small buffers");
    if (!direct) {
      GS_TRY(grow_pair<int32_t>(nullptr, &sb->h_rp, &sb->cap_hrows, rows), "small buffers");
      GS_TRY(grow_pair<int32_t>(nullptr, &sb->h_ci, &sb->cap_hnnz, nnz), "small buffers");
    }
    if ((size_t)G + 1 > sb->cap_g || !sb->d_voff) {
      size_t c1 = 0;
      const size_t need = (size_t)G + 1;
      sb->cap_g = 0;  // until all of them hold it: a failure below leaves some without memory
      GS_TRY(grow_pair(&sb->d_voff, &sb->h_voff, &c1, need), "small buffers");
      c1 = 0; GS_TRY(grow_pair(&sb->d_eoff, &sb->h_eoff, &c1, need), "small buffers");
      c1 = 0; GS_TRY(grow_pair(&sb->d_gm, &sb->h_gm, &c1, need), "small buffers");
      c1 = 0; GS_TRY(grow_pair(&sb->d_gn, &sb->h_gn, &c1, need), "small buffers");
      c1 = 0; GS_TRY(grow_pair<unsigned long long>(&sb->d_sums, nullptr, &c1, kSmallSums * need), "small buffers");
      c1 = 0; GS_TRY(grow_pair<unsigned long long>(&sb->d_csum, nullptr, &c1, 26 * need), "small buffers");
      c1 = 0; GS_TRY(grow_pair<unsigned long long>(&sb->d_x, nullptr, &c1, 34 * need), "small buffers");
      if (!sb->d_misc) GS_TRY(cudaMalloc(&sb->d_misc, sizeof(int32_t) * (kSmallClasses + 1)), "small buffers");
      cg = c1 / 34;
    }
    sb->cap_g = cg;
  }
  int32_t class_off[kSmallClasses + 1] = {0};
  std::vector<int2> units;
  {
    std::vector<int32_t> gn((size_t)G);
    std::vector<int64_t> gm((size_t)G);
    for (int32_t gi = 0; gi < G; ++gi) {
      gn[(size_t)gi] = graphs[gi]->n;
      gm[(size_t)gi] = graphs[gi]->m;
    }
    small_units(gn, gm, &units, class_off);
    GS_TRY(grow_pair(&sb->d_units, &sb->h_units, &sb->cap_units, units.size()), "small buffers");
    std::memcpy(sb->h_units, units.data(), sizeof(int2) * units.size());
  }
  if (!sb->fork.start) {
    GS_TRY(cudaEventCreateWithFlags(&sb->fork.start, cudaEventDisableTiming), "small fork");
    for (int c = 0; c < kSmallClasses; ++c) {
      GS_TRY(cudaEventCreateWithFlags(&sb->fork.done[c], cudaEventDisableTiming), "small fork");
      GS_TRY(cudaStreamCreateWithFlags(&sb->fork.stream[c], cudaStreamNonBlocking), "small fork");
    }
  }
  std::memcpy(sb->h_voff, voff.data(), sizeof(int64_t) * voff.size());
  std::memcpy(sb->h_eoff, eoff.data(), sizeof(int64_t) * eoff.size());
  for (int32_t gi = 0; gi < G; ++gi) {
    sb->h_gn[gi] = graphs[gi]->n;
    sb->h_gm[gi] = graphs[gi]->m;
  }
  if (!direct) {  // CSR packed on the host cores, each thread the graphs whose entries start in its share
    const int nt = (int)std::max<int64_t>(1, std::min<int64_t>(host_threads(), eoff[G] >> 16));
    host_run(nt, [&](int t) {
      const int64_t e0 = eoff[G] * t / nt, e1 = eoff[G] * (t + 1) / nt;
      int32_t gi = t == 0 ? 0 : (int32_t)(std::lower_bound(eoff.begin(), eoff.begin() + G, e0) - eoff.begin());
      for (; gi < G && (eoff[gi] < e1 || t == nt - 1); ++gi) {
        std::memcpy(sb->h_rp + voff[gi], graphs[gi]->rp, sizeof(int32_t) * (graphs[gi]->n + 1));
        if (graphs[gi]->m > 0)
          std::memcpy(sb->h_ci + eoff[gi], graphs[gi]->ci, sizeof(int32_t) * 2 * graphs[gi]->m);
      }
    });
  }
  const int32_t* src_rp = direct ? graphs[0]->rp : sb->h_rp;
  const int32_t* src_ci = direct ? graphs[0]->ci : sb->h_ci;
  const bool graph_mode = cfg.use_graph != 0;
  // the sequence; returns the first failure (for a capture, the capture is
  // ended by the caller)
  auto issue = [&]() -> cudaError_t {
    cudaError_t r = cudaSuccess;
    const size_t b4 = sizeof(int32_t), b8 = sizeof(int64_t);
    r = cudaMemcpyAsync(sb->d_rp, src_rp, b4 * rows, cudaMemcpyHostToDevice, s);
    if (r == cudaSuccess && eoff[G] > 0) r = cudaMemcpyAsync(sb->d_ci, src_ci, b4 * (size_t)eoff[G], cudaMemcpyHostToDevice, s);
    if (r == cudaSuccess) r = cudaMemcpyAsync(sb->d_voff, sb->h_voff, b8 * (G + 1), cudaMemcpyHostToDevice, s);
    if (r == cudaSuccess) r = cudaMemcpyAsync(sb->d_eoff, sb->h_eoff, b8 * (G + 1), cudaMemcpyHostToDevice, s);
    if (r == cudaSuccess) r = cudaMemcpyAsync(sb->d_gn, sb->h_gn, b4 * G, cudaMemcpyHostToDevice, s);
    if (r == cudaSuccess) r = cudaMemcpyAsync(sb->d_gm, sb->h_gm, b8 * G, cudaMemcpyHostToDevice, s);
    if (r == cudaSuccess)
      r = cudaMemcpyAsync(sb->d_units, sb->h_units, sizeof(int2) * units.size(), cudaMemcpyHostToDevice, s);
    if (r == cudaSuccess) r = cudaMemsetAsync(sb->d_misc, 0, b4 * (kSmallClasses + 1), s);
    if (r == cudaSuccess) r = cudaMemsetAsync(sb->d_sums, 0, sizeof(unsigned long long) * kSmallSums * (size_t)G, s);
    if (r != cudaSuccess) return r;
    const SmallGraphs sg = {G,           sb->d_rp,    sb->d_ci,   sb->d_gn,   sb->d_voff, sb->d_eoff, sb->d_gm,
                            sb->d_units, sb->d_misc, sb->d_misc + kSmallClasses, sb->d_sums, sb->d_csum};
    // eager launches time each class, one after the other
    if (run_small_graphs(sg, class_off, cfg, graph_mode ? nullptr : L->ev + kEvSmall0,
                         graph_mode ? &sb->fork : nullptr, s) != GC_OK)
      return cudaErrorLaunchFailure;
    DevGraph dg = DevGraph();
    dg.G = G;
    dg.gn = sb->d_gn;
    dg.gm = sb->d_gm;
    if (run_derive(dg, sb->d_csum, sb->d_x, sb->d_misc + kSmallClasses, s) != GC_OK) return cudaErrorLaunchFailure;
    r = cudaMemcpyAsync(h_x_dst, sb->d_x, sizeof(unsigned long long) * (size_t)G * 34, cudaMemcpyDeviceToHost, s);
    if (r == cudaSuccess) r = cudaMemcpyAsync(L->h_status, sb->d_misc + kSmallClasses, b4, cudaMemcpyDeviceToHost, s);
    return r;
  };
  GS_TRY(cudaEventRecord(L->ev[kEvSmallSeq0], s), "small event");
  if (graph_mode) {
    cudaGraph_t graph = nullptr;
    GS_TRY(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal), "capture small-graph launch");
    const cudaError_t r = issue();
    const cudaError_t r2 = cudaStreamEndCapture(s, &graph);
    if (r != cudaSuccess || r2 != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      GS_TRY(r != cudaSuccess ? r : r2, "capture small-graph launch");
    }
    if (sb->exec) {
      cudaGraphExecUpdateResultInfo info;
      if (cudaGraphExecUpdate(sb->exec, graph, &info) != cudaSuccess) {
        cudaGetLastError();
        cudaGraphExecDestroy(sb->exec);
        sb->exec = nullptr;
      }
    }
    if (!sb->exec) {
      e = cudaGraphInstantiate(&sb->exec, graph, 0);
      if (e != cudaSuccess) {
        cudaGraphDestroy(graph);
        sb->exec = nullptr;
        GS_TRY(e, "instantiate small-graph launch");
      }
    }
    cudaGraphDestroy(graph);
    GS_TRY(cudaGraphLaunch(sb->exec, s), "replay small-graph launch");
    L->replayed = true;
  } else {
    GS_TRY(issue(), "small-graph launch");
    L->timed_classes = true;
  }
  GS_TRY(cudaEventRecord(L->ev[kEvSmallSeq1], s), "small event");
  GS_TRY(cudaEventRecord(sb->busy, s), "small event");
  L->timed_small = true;
#undef GS_TRY
  return GC_OK;
}

// Counts `graphs` as one launch on `s`: small graphs on the bitmatrix kernels,
// the others as one disjoint union. Results land in L->h_x when L->done
// completes. Runs in the dispatcher thread (or the flushing thread in manual
// mode) without holding the batch lock.
void run_launch(gc_batch b, std::vector<PendingGraph>& graphs, cudaStream_t s, Launch* L) {
  const BatchConfig cfg = L->cfg;
  auto is_small = [&](const PendingGraph& pg) {
    return pg.n <= cfg.small_n_max && small_class_of(pg.n) < kSmallClasses;
  };
  std::vector<PendingGraph*> small, large;
  for (auto& pg : graphs) (is_small(pg) ? small : large).push_back(&pg);
  L->slot.resize(graphs.size());
  {
    int32_t is = 0, il = (int32_t)small.size();
    for (size_t k = 0; k < graphs.size(); ++k) L->slot[k] = is_small(graphs[k]) ? is++ : il++;
  }
  gc_status st = GC_OK;
  L->h_status[0] = 0;
  L->h_status[1] = 0;
  if (!small.empty()) st = run_small(small, s, L, L->h_x, &b->small[L->stream_slot], cfg);
  if (st == GC_OK && !large.empty()) {
    cudaEventRecord(L->ev[kEvUnion0], s);
    ForkSet*& fs = b->forks[L->stream_slot];
    if (!fs) fs = fork_acquire(b->device, 0);  // the slots' streams have the default priority
    if (!fs) {
      st = GC_ERR_CUDA;
      L->error = gc_last_error();
    } else {
      st = run_union(large, s, fs, L, L->h_x + 34 * small.size(), L->h_status + 1);
    }
    cudaEventRecord(L->ev[kEvUnion1], s);
    L->timed_union = st == GC_OK;
  }
  L->launch_status = st;
  if (st != GC_OK) cudaStreamSynchronize(s);  // copies already queued read the launch's host blocks
  if (st == GC_OK) {
    cudaError_t e = cudaEventRecord(L->done, s);
    if (e != cudaSuccess) {
      L->launch_status = cuda_fail(e, "batch event");
      L->error = gc_last_error();
      cudaStreamSynchronize(s);  // no event tells when the launch's buffers are free
    }
  }
}

void free_launch(Launch* L) {
  if (L->h_x) cudaFreeHost(L->h_x);
  if (L->h_status) cudaFreeHost(L->h_status);
  if (L->done) cudaEventDestroy(L->done);
  for (auto& ev : L->ev)
    if (ev) cudaEventDestroy(ev);
  delete L;
}

// Events and pinned results of a launch of G graphs (a spare launch keeps its
// own).
cudaError_t init_launch(Launch* L, size_t G) {
  cudaError_t e = cudaSuccess;
  if (G > L->cap_x) {
    if (L->h_x) cudaFreeHost(L->h_x);
    L->h_x = nullptr;
    L->cap_x = 0;
    const size_t want = G + G / 4 + 16;
    e = cudaMallocHost(&L->h_x, sizeof(unsigned long long) * 34 * want);
    if (e == cudaSuccess) L->cap_x = want;
  }
  if (e == cudaSuccess && !L->h_status) e = cudaMallocHost(&L->h_status, 2 * sizeof(int32_t));
  if (e == cudaSuccess && !L->done) e = cudaEventCreateWithFlags(&L->done, cudaEventDisableTiming);
  for (auto& ev : L->ev)
    if (e == cudaSuccess && !ev) e = cudaEventCreate(&ev);
  return e;
}

// Must hold b->mu.
void retire_locked(gc_batch b) {
  for (size_t i = 0; i < b->inflight.size();) {
    Launch* L = b->inflight[i];
    bool finished = L->launch_status != GC_OK;
    if (!finished) {
      cudaError_t q = cudaEventQuery(L->done);
      if (q == cudaErrorNotReady) {
        ++i;
        continue;
      }
      if (q != cudaSuccess) {
        L->launch_status = cuda_fail(q, "batch launch");
        L->error = gc_last_error();
        cudaStreamSynchronize(L->stream);  // whatever it was, the GPU must be done with the launch's buffers
      }
    }
    if (L->launch_status == GC_OK) {  // device times of the launch
      auto ms = [&](int a, int z) {
        float f = 0.f;
        return cudaEventElapsedTime(&f, L->ev[a], L->ev[z]) == cudaSuccess ? (double)f : 0.0;
      };
      for (int c = 0; c < kSmallClasses; ++c)
        b->last_stats[c] = L->timed_classes ? ms(kEvSmall0 + 2 * c, kEvSmall0 + 2 * c + 1) : 0.0;
      b->last_stats[kSmallClasses] = L->timed_small ? ms(kEvSmallSeq0, kEvSmallSeq1) : 0.0;
      b->last_stats[kSmallClasses + 1] = L->timed_union ? ms(kEvUnion0, kEvUnion1) : 0.0;
      b->last_stats[kSmallClasses + 2] = L->replayed ? 1.0 : 0.0;
      cudaGetLastError();
    }
    std::shared_ptr<Results> out;
    gc_status status = L->launch_status;
    if (status == GC_OK && (L->h_status[0] | L->h_status[1])) status = GC_ERR_CUDA;
    if (status == GC_OK) {
      try {
        out = std::make_shared<Results>(L->h_x, L->h_x + 34 * L->tickets.size());
      } catch (...) {
        status = GC_ERR_NOMEM;
      }
    }
    for (size_t k = 0; k < L->tickets.size(); ++k) {
      Ticket* t = b->find(L->tickets[k]);  // live until polled
      t->state = Ticket::kDone;
      t->status = status;
      t->slot = L->slot.size() > k ? L->slot[k] : 0;
      t->out = out;
    }
    b->in_use -= L->bytes;
    L->owners.clear();
    try {
      b->spare.push_back(L);
    } catch (...) {
      free_launch(L);
    }
    b->inflight.erase(b->inflight.begin() + i);
    b->cv.notify_all();
  }
}

// Whether the batch has nothing to do. Must hold b->mu.
bool idle(gc_batch b) { return b->pending.empty() && b->inflight.empty(); }

// Gives back the pinned memory kept beyond the limits. Freeing it waits for the
// whole device, so no lock is held and the batch is idle.
void trim(gc_batch b) {
  for (;;) {
    Launch* L = nullptr;
    {
      std::lock_guard<std::mutex> lk(b->mu);
      if (b->spare.size() <= kMaxSpare) break;
      L = b->spare.back();
      b->spare.pop_back();
    }
    free_launch(L);
  }
  b->host->trim();
}

// Takes every pending graph (up to the int32 edge limit) and launches it.
// Called without the lock; returns false if nothing was pending.
bool launch_pending(gc_batch b) {
  std::vector<PendingGraph> take;
  Launch* L = nullptr;
  {
    std::lock_guard<std::mutex> lk(b->mu);
    if (b->pending.empty()) return false;
    if (!b->spare.empty()) {
      L = b->spare.back();
      b->spare.pop_back();
    } else {
      b->spare.reserve(b->spare.size() + kMaxSpare);  // a launch can always be put back
      L = new Launch();
    }
    L->tickets.clear();
    L->slot.clear();
    L->bytes = 0;
    L->timed_classes = L->timed_small = L->timed_union = L->replayed = false;
    L->launch_status = GC_OK;
    L->error.clear();
    int64_t nnz = 0, nv = 0;
    try {  // from here to the launch nothing may throw: a graph taken from the queue must reach its ticket
      const size_t most = b->pending.size();
      take.reserve(most);
      L->tickets.reserve(most);
      L->owners.reserve(most);
      L->slot.reserve(most);
      b->inflight.reserve(b->inflight.size() + 1 + kMaxInflight);
    } catch (...) {
      b->spare.push_back(L);  // where it was, or the place of one that was
      throw;
    }
    while (!b->pending.empty()) {
      PendingGraph& pg = b->pending.front();
      if (!take.empty() && (nnz + 2 * pg.m >= (1LL << 31) - 1 || nv + pg.n >= (1LL << 31) - 1)) break;
      nnz += 2 * pg.m;
      nv += pg.n;
      L->tickets.push_back(pg.ticket);
      L->bytes += pg.bytes;
      if (pg.owner && (L->owners.empty() || L->owners.back() != pg.owner)) L->owners.push_back(pg.owner);
      take.push_back(std::move(pg));
      b->pending.pop_front();
    }
    // a stream slot no launch in flight holds (the dispatcher keeps fewer
    // than max_inflight launches in flight); manual flushes take the slots in
    // turn (a slot's buffers wait for their previous use)
    int slot = -1;
    for (int k = 0; k < b->cfg.max_inflight && slot < 0; ++k) {
      bool used = false;
      for (Launch* o : b->inflight) used |= o->stream_slot == k;
      if (!used) slot = k;
    }
    if (slot < 0) {
      slot = b->next_stream % b->cfg.max_inflight;
      b->next_stream = slot + 1;
    }
    L->stream_slot = slot;
    L->cfg = b->cfg;
    L->stream = b->streams[slot];
  }
  cudaSetDevice(b->device);
  if (init_launch(L, take.size()) != cudaSuccess) {
    cudaGetLastError();
    L->launch_status = GC_ERR_NOMEM;
  } else {
    try {
      run_launch(b, take, L->stream, L);
    } catch (...) {
      L->launch_status = no_memory();
      cudaStreamSynchronize(L->stream);  // what was queued reads the launch's host blocks
    }
  }
  {
    std::lock_guard<std::mutex> lk(b->mu);
    b->inflight.push_back(L);
    b->cv.notify_all();
  }
  return true;
}

void dispatcher_main(gc_batch b) {
  OutsideCapture relaxed;
  cudaSetDevice(b->device);
  std::unique_lock<std::mutex> lk(b->mu);
  bool trimmed = true;  // since the batch was last busy
  while (!b->stop) {
    retire_locked(b);
    if (!idle(b)) {
      trimmed = false;
    } else if (!trimmed) {
      trimmed = true;
      lk.unlock();
      trim(b);
      lk.lock();
      continue;
    }
    if (!b->pending.empty() && (int)b->inflight.size() < b->cfg.max_inflight) {
      lk.unlock();
      try {
        launch_pending(b);
      } catch (...) {  // no memory for the launch's lists: the graphs are still pending
        std::this_thread::sleep_for(std::chrono::milliseconds(1));
      }
      lk.lock();
      continue;
    }
    // woken by a submission; launches in flight are looked at now and then
    if (b->inflight.empty()) b->cv.wait_for(lk, std::chrono::milliseconds(1));
    else b->cv.wait_for(lk, std::chrono::microseconds(20));
  }
}

// One turn of a poll's wait, with b->mu held by lk: the first turns only give
// way to other threads (a small launch takes a fraction of a millisecond), the
// later ones sleep.
void poll_wait(gc_batch b, std::unique_lock<std::mutex>* lk, std::chrono::steady_clock::time_point began) {
  if (std::chrono::steady_clock::now() - began < std::chrono::microseconds(500)) {
    lk->unlock();
    std::this_thread::yield();
    lk->lock();
  } else {
    b->cv.wait_for(*lk, std::chrono::microseconds(50));
  }
}

}  // namespace

// Gives back what the checks hold that the GPU is done with (all: waits for them).
static void reclaim_checks(gc_batch b, bool all) {
  for (Check& c : b->checks) {
    if (!c.busy || !c.own) continue;  // free, or its submission still looks at it
    if (all) cudaEventSynchronize(c.done);
    else if (cudaEventQuery(c.done) == cudaErrorNotReady) continue;
    cudaGetLastError();
    if (c.d) cudaFreeAsync(c.d, c.stream);
    c.d = nullptr;
    c.own.reset();
    c.busy = false;
  }
}

// Whether the graph copied to `own` (row pointers, then columns; pinned) passes
// every check of validate_csr, by k_check_csr; its row pointers have been
// checked. false also when a device step fails, when the checks are all busy, or
// when the GPU has no room for the check in time: the caller then asks the host.
// Neither priority nor anything else takes a running CTA's place, so that behind
// kernels that fill the GPU a check would last as long as they do: a submission
// gives it 0.3 ms and 0.5 ns an entry (3.5M entries take 0.9 ms on an idle GPU, the
// host's checks 6.2), and leaves what it holds to a later one.
static bool checked_on_device(gc_batch b, int32_t n, int32_t nnz, const std::shared_ptr<HostBlock>& own) {
  OutsideCapture relaxed;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || (dev != b->device && cudaSetDevice(b->device) != cudaSuccess)) {
    cudaGetLastError();
    return false;
  }
  Check* c = nullptr;
  {
    std::lock_guard<std::mutex> lk(b->check_mu);
    reclaim_checks(b, false);
    for (Check& k : b->checks)
      if (!k.busy) {
        c = &k;
        c->busy = true;
        break;
      }
  }
  bool ok = false, left = false;
  if (c) {
    cudaError_t e = cudaSuccess;
    if (!c->stream) {
      int least = 0, greatest = 0;
      e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
      if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&c->stream, cudaStreamNonBlocking, greatest);
    }
    if (e == cudaSuccess && !c->done) e = cudaEventCreateWithFlags(&c->done, cudaEventDisableTiming);
    if (e == cudaSuccess && !c->bad) e = cudaMallocHost(&c->bad, sizeof(int32_t));
    const size_t words = (size_t)n + 1 + (size_t)nnz;
    bool queued = false;
    if (e == cudaSuccess && (e = pool_alloc(&c->d, sizeof(int32_t) * (words + 1), c->stream)) == cudaSuccess) {
      queued = true;
      e = cudaMemsetAsync(c->d, 0, sizeof(int32_t), c->stream);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->d + 1, own->p, sizeof(int32_t) * words, cudaMemcpyHostToDevice, c->stream);
      if (e == cudaSuccess) {
        const int64_t blocks = ((int64_t)nnz + 255) / 256;
        k_check_csr<<<(int)std::min<int64_t>(blocks, 8LL * (count_grid_size() / kCtasPerSm)), 256, 0, c->stream>>>(
            n, nnz, c->d + 1, c->d + 1 + n + 1, c->d);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess) e = cudaMemcpyAsync(c->bad, c->d, sizeof(int32_t), cudaMemcpyDeviceToHost, c->stream);
      if (e == cudaSuccess) e = cudaEventRecord(c->done, c->stream);
    }
    if (e == cudaSuccess) {
      const auto until = std::chrono::steady_clock::now() + std::chrono::nanoseconds(300000 + (int64_t)nnz / 2);
      while ((e = cudaEventQuery(c->done)) == cudaErrorNotReady && std::chrono::steady_clock::now() < until)
        std::this_thread::yield();
      left = e == cudaErrorNotReady;
      ok = e == cudaSuccess && *c->bad == 0;
    }
    if (queued && !left && e != cudaSuccess) cudaStreamSynchronize(c->stream);  // `own` may be read
    if (e != cudaSuccess) cudaGetLastError();
    std::lock_guard<std::mutex> lk(b->check_mu);
    if (left) {
      c->own = own;  // busy until reclaimed
    } else {
      if (c->d) cudaFreeAsync(c->d, c->stream);
      c->d = nullptr;
      c->busy = false;
    }
  }
  if (dev != b->device) cudaSetDevice(dev);
  return ok;
}

extern "C" {

gc_status gc_batch_create(int64_t device_mem_budget_bytes, uint32_t flags, gc_batch* out) try {
  if (!out) { set_error("out is NULL"); return GC_ERR_ARG; }
  *out = nullptr;
  if (device_mem_budget_bytes <= 0 || (flags & ~GC_BATCH_MANUAL)) {
    set_error("bad budget or flags");
    return GC_ERR_ARG;
  }
  gc_batch b = new (std::nothrow) gc_batch_s();
  if (!b) { set_error("host allocation failed"); return GC_ERR_NOMEM; }
  b->budget = device_mem_budget_bytes;
  b->flags = flags;
  cudaGetDevice(&b->device);
  for (auto& s : b->streams) {
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      gc_status st = cuda_fail(e, "batch stream");
      for (auto& t : b->streams)
        if (t) cudaStreamDestroy(t);
      delete b;
      return st;
    }
  }
  count_grid_size();
  gc_status st = small_graphs_setup();
  if (st != GC_OK) {
    for (auto& t : b->streams) cudaStreamDestroy(t);
    delete b;
    return st;
  }
  load_tuned_config(&b->cfg, nullptr);
  try {
    if (!(flags & GC_BATCH_MANUAL)) b->dispatcher = std::thread(dispatcher_main, b);
  } catch (...) {
    for (auto& t : b->streams) cudaStreamDestroy(t);
    delete b;
    set_error("the dispatcher thread could not be started");
    return GC_ERR_NOMEM;
  }
  *out = b;
  return GC_OK;
} catch (...) {
  return no_memory();
}

gc_status gc_batch_set_param(gc_batch b, int32_t param, int32_t value) {
  if (!b) { set_error("batch is NULL"); return GC_ERR_ARG; }
  std::lock_guard<std::mutex> lk(b->mu);
  if (param == GC_PARAM_SMALL_N_MAX) {
    if (value < 0 || value > kSmallClassN[kSmallClasses - 1]) { set_error("small_n_max outside [0, 1024]"); return GC_ERR_ARG; }
    b->cfg.small_n_max = value;
  } else if (param >= GC_PARAM_BLOCK_N64 && param < GC_PARAM_BLOCK_N64 + kSmallClasses) {
    if (value != 64 && value != 128 && value != 256 && value != 512) { set_error("block must be 64, 128, 256 or 512"); return GC_ERR_ARG; }
    b->cfg.class_block[param - GC_PARAM_BLOCK_N64] = value;
  } else if (param == GC_PARAM_USE_GRAPH) {
    if (value != 0 && value != 1) { set_error("use_graph must be 0 or 1"); return GC_ERR_ARG; }
    b->cfg.use_graph = value;
  } else if (param == GC_PARAM_MAX_INFLIGHT) {
    if (value < 1 || value > kMaxInflight) { set_error("max_inflight must be 1 .. 4"); return GC_ERR_ARG; }
    b->cfg.max_inflight = value;
  } else {
    set_error("unknown parameter");
    return GC_ERR_ARG;
  }
  return GC_OK;
}

gc_status gc_batch_get_param(gc_batch b, int32_t param, int32_t* value) {
  if (!b || !value) { set_error("NULL argument"); return GC_ERR_ARG; }
  std::lock_guard<std::mutex> lk(b->mu);
  if (param == GC_PARAM_SMALL_N_MAX) *value = b->cfg.small_n_max;
  else if (param >= GC_PARAM_BLOCK_N64 && param < GC_PARAM_BLOCK_N64 + kSmallClasses)
    *value = b->cfg.class_block[param - GC_PARAM_BLOCK_N64];
  else if (param == GC_PARAM_USE_GRAPH) *value = b->cfg.use_graph;
  else if (param == GC_PARAM_MAX_INFLIGHT) *value = b->cfg.max_inflight;
  else { set_error("unknown parameter"); return GC_ERR_ARG; }
  return GC_OK;
}

gc_status gc_batch_last_stats(gc_batch b, double* out) {
  if (!b || !out) { set_error("NULL argument"); return GC_ERR_ARG; }
  std::lock_guard<std::mutex> lk(b->mu);
  for (int i = 0; i < GC_BATCH_STATS; ++i) out[i] = b->last_stats[i];
  return GC_OK;
}

gc_status gc_batch_submit(gc_batch b, int32_t n, const int32_t* row_ptr, const int32_t* col_idx,
                          uint64_t* ticket_out) try {
  if (!b || !ticket_out || !row_ptr || n < 0) { set_error("bad arguments"); return GC_ERR_ARG; }
  // Graphs of kDeviceCheck entries or more are checked on the device, from the
  // copy, once their row pointers have been checked; what fails there (or
  // cannot be checked there) gets the host's checks, for the code and message.
  constexpr int32_t kDeviceCheck = 1 << 16;
  bool on_device = n > 0 && row_ptr[0] == 0 && row_ptr[n] >= kDeviceCheck && row_ptr[n] % 2 == 0 && col_idx;
  if (on_device) {
    bool ascending = true;
    for (int32_t x = 0; x < n; ++x) ascending &= row_ptr[x + 1] >= row_ptr[x];
    on_device = ascending;
  }
  gc_status st = GC_OK;
  if (!on_device && (st = validate_csr(n, row_ptr, col_idx)) != GC_OK) return st;
  const int64_t m = row_ptr[n] / 2;
  const int64_t bytes = footprint(n, m);
  // Its share of the budget first, so that a graph that does not fit now costs
  // neither a copy nor device memory for the check. An invalid graph is refused as
  // such all the same, by the host's checks.
  if (!b->reserve(bytes)) {
    if (on_device && (st = validate_csr(n, row_ptr, col_idx)) != GC_OK) return st;
    if (bytes > b->budget) {
      set_error("graph needs more device memory than the whole budget");
      return GC_ERR_NOMEM;
    }
    set_error("device-memory budget is full");
    return GC_ERR_BUSY;
  }
  struct Reserved {  // given back unless the graph is admitted
    gc_batch b;
    int64_t bytes;
    ~Reserved() {
      if (bytes) b->release(bytes);
    }
  } reserved = {b, bytes};
  PendingGraph pg;
  pg.n = n;
  pg.m = m;
  pg.bytes = bytes;
  try {
    pg.owner = host_block(b->host, (size_t)n + 1 + 2 * (size_t)m);
    int32_t* own = pg.owner->p;
    pg.rp = own;
    pg.ci = own + n + 1;
    std::memcpy(own, row_ptr, sizeof(int32_t) * ((size_t)n + 1));
    const int nt = (int)std::max<int64_t>(1, std::min<int64_t>(host_threads(), 2 * m >> 18));
    host_run(nt, [&](int t) {
      const size_t e0 = 2 * (size_t)m * (size_t)t / (size_t)nt, e1 = 2 * (size_t)m * ((size_t)t + 1) / (size_t)nt;
      if (e1 > e0) std::memcpy(own + n + 1 + e0, col_idx + e0, sizeof(int32_t) * (e1 - e0));
    });
  } catch (...) {
    set_error("host allocation failed");
    return GC_ERR_NOMEM;
  }
  if (on_device && !(pg.owner->pinned && checked_on_device(b, n, row_ptr[n], pg.owner)) &&
      (st = validate_csr(n, pg.rp, pg.ci)) != GC_OK)
    return st;
  {
    std::lock_guard<std::mutex> lk(b->mu);
    pg.ticket = b->admit();
    *ticket_out = pg.ticket;
    b->pending.back() = std::move(pg);
    reserved.bytes = 0;  // the launch's retirement gives it back
  }
  b->cv.notify_all();
  return GC_OK;
} catch (...) {
  return no_memory();
}

gc_status gc_batch_submit_many(gc_batch b, int64_t G, const int32_t* nvert, const int64_t* voff, const int64_t* eoff,
                               const int32_t* row_ptr, const int32_t* col_idx, uint64_t* tickets_out) try {
  if (!b || G < 0 || (G > 0 && (!nvert || !voff || !eoff || !row_ptr || !tickets_out))) {
    set_error("bad arguments");
    return GC_ERR_ARG;
  }
  if (G == 0) return GC_OK;
  // the library's copy: one buffer for all graphs, rows then columns, each
  // graph at its own offset (own_v, own_e), filled while validating
  std::vector<int64_t> own_v((size_t)G + 1), own_e((size_t)G + 1);
  own_v[0] = own_e[0] = 0;
  for (int64_t g = 0; g < G; ++g) {
    const int32_t n = nvert[g];
    if (n < 0 || eoff[g + 1] < eoff[g]) {
      set_error("graph " + std::to_string(g) + ": negative size or decreasing offsets");
      return GC_ERR_ARG;
    }
    own_v[g + 1] = own_v[g] + n + 1;
    own_e[g + 1] = own_e[g] + (eoff[g + 1] - eoff[g]);
  }
  std::shared_ptr<HostBlock> owner;
  try {
    owner = host_block(b->host, (size_t)(own_v[G] + own_e[G]));
  } catch (...) {
    set_error("host allocation failed");
    return GC_ERR_NOMEM;
  }
  int32_t* own_rp = owner->p;
  int32_t* own_ci = owner->p + own_v[G];
  std::vector<PendingGraph> pgs((size_t)G);
  // shares of about equal entries, at least 2^14 each, four to a thread
  const int nt = (int)std::max<int64_t>(1, std::min<int64_t>({4 * (int64_t)host_threads(), G, own_e[G] >> 14}));
  std::vector<gc_status> res(nt, GC_OK);
  std::vector<std::string> msg(nt);
  auto work = [&](int t) {  // the graphs whose entries start in this thread's share
    std::vector<int32_t> fill;  // symmetry-walk scratch of this thread
    const int64_t e0 = own_e[G] * t / nt, e1 = own_e[G] * (t + 1) / nt;
    int64_t g = t == 0 ? 0 : std::lower_bound(own_e.begin(), own_e.begin() + G, e0) - own_e.begin();
    for (; g < G && (own_e[g] < e1 || t == nt - 1); ++g) {
      const int32_t n = nvert[g];
      const int32_t* rp = row_ptr + voff[g];
      const int32_t* ci = col_idx ? col_idx + eoff[g] : nullptr;
      if ((int64_t)rp[n] != eoff[g + 1] - eoff[g]) {
        res[t] = GC_ERR_ARG;
        msg[t] = "graph " + std::to_string(g) + ": offsets disagree with row_ptr";
        return;
      }
      gc_status st = (int64_t)rp[n] < (1 << 20) ? validate_csr_small(n, rp, ci, &fill) : validate_csr(n, rp, ci);
      if (st != GC_OK) {
        res[t] = st;
        msg[t] = "graph " + std::to_string(g) + ": " + gc_last_error();
        return;
      }
      PendingGraph& pg = pgs[(size_t)g];
      pg.n = n;
      pg.m = rp[n] / 2;
      pg.bytes = footprint(n, pg.m);
      std::memcpy(own_rp + own_v[g], rp, sizeof(int32_t) * ((size_t)n + 1));
      if (pg.m > 0) std::memcpy(own_ci + own_e[g], ci, sizeof(int32_t) * 2 * (size_t)pg.m);
      pg.rp = own_rp + own_v[g];
      pg.ci = own_ci + own_e[g];
      pg.owner = owner;
    }
  };
  try {
    host_run(nt, work);
  } catch (...) {
    set_error("host allocation failed");
    return GC_ERR_NOMEM;
  }
  for (int t = 0; t < nt; ++t)
    if (res[t] != GC_OK) {
      set_error(msg[t]);
      return res[t];
    }
  int64_t bytes = 0;
  for (auto& pg : pgs) bytes += pg.bytes;
  {
    std::lock_guard<std::mutex> lk(b->mu);
    if (bytes > b->budget) {
      set_error("graphs need more device memory than the whole budget");
      return GC_ERR_NOMEM;
    }
    if (b->in_use + bytes > b->budget) {
      set_error("device-memory budget is full");
      return GC_ERR_BUSY;
    }
    int64_t g = 0;
    try {
      for (; g < G; ++g) {
        pgs[(size_t)g].ticket = b->admit();
        tickets_out[g] = pgs[(size_t)g].ticket;
        b->pending.back() = std::move(pgs[(size_t)g]);
      }
    } catch (...) {  // all or none
      for (; g > 0; --g) b->dismiss();
      throw;
    }
    b->in_use += bytes;
  }
  b->cv.notify_all();
  return GC_OK;
} catch (...) {
  return no_memory();
}

gc_status gc_batch_flush(gc_batch b) try {
  if (!b) { set_error("batch is NULL"); return GC_ERR_ARG; }
  if (b->flags & GC_BATCH_MANUAL) {
    OutsideCapture relaxed;
    while (launch_pending(b)) {
    }
  } else {
    b->cv.notify_all();
  }
  return GC_OK;
} catch (...) {
  return no_memory();
}

gc_status gc_batch_poll(gc_batch b, uint64_t ticket, uint64_t* global_out, uint64_t* global_hi,
                        int32_t timeout_us) try {
  if (!b || !global_out) { set_error("NULL argument"); return GC_ERR_ARG; }
  OutsideCapture relaxed;
  const auto began = std::chrono::steady_clock::now();
  const auto deadline = began + std::chrono::microseconds(timeout_us > 0 ? timeout_us : 0);
  std::unique_lock<std::mutex> lk(b->mu);
  for (;;) {
    Ticket* t = b->find(ticket);
    if (!t) {
      set_error("unknown or retired ticket");
      return GC_ERR_ARG;
    }
    if (b->flags & GC_BATCH_MANUAL) retire_locked(b);
    if (t->state == Ticket::kDone) {
      const Ticket r = std::move(*t);
      b->retire(ticket);
      b->drop_retired();
      const bool rest = (b->flags & GC_BATCH_MANUAL) && idle(b);
      lk.unlock();
      if (rest) trim(b);  // otherwise the dispatcher's
      if (r.status != GC_OK) {
        set_error("batch launch failed");
        return r.status;
      }
      const uint64_t* x = r.out->data() + 34 * (size_t)r.slot;
      bool need_hi = false;
      for (int i = 0; i < 17; ++i) {
        global_out[i] = x[2 * i];
        if (global_hi) global_hi[i] = x[2 * i + 1];
        if (x[2 * i + 1]) need_hi = true;
      }
      if (need_hi && !global_hi) {
        set_error("a global count exceeds 64 bits and global_hi is NULL");
        return GC_ERR_OVERFLOW;
      }
      return GC_OK;
    }
    if (timeout_us == 0) return GC_PENDING;
    if (timeout_us > 0 && std::chrono::steady_clock::now() >= deadline) return GC_PENDING;
    poll_wait(b, &lk, began);
  }
} catch (...) {
  return no_memory();
}

gc_status gc_batch_poll_many(gc_batch b, int64_t G, const uint64_t* tickets, uint64_t* global_out,
                             uint64_t* global_hi, int32_t timeout_us) try {
  if (!b || G < 0 || (G > 0 && (!tickets || !global_out))) { set_error("bad arguments"); return GC_ERR_ARG; }
  OutsideCapture relaxed;
  const auto began = std::chrono::steady_clock::now();
  const auto deadline = began + std::chrono::microseconds(timeout_us > 0 ? timeout_us : 0);
  std::unique_lock<std::mutex> lk(b->mu);
  for (int64_t i = 0; i < G; ++i)
    if (!b->find(tickets[i])) {
      set_error("ticket " + std::to_string(i) + " is unknown or retired");
      return GC_ERR_ARG;
    }
  int64_t ready = 0;  // tickets[0 .. ready) are known to be done
  for (;;) {
    if (b->flags & GC_BATCH_MANUAL) retire_locked(b);
    for (; ready < G; ++ready) {
      const Ticket* t = b->find(tickets[ready]);
      if (!t) {  // retired by another thread's poll meanwhile
        set_error("ticket " + std::to_string(ready) + " is unknown or retired");
        return GC_ERR_ARG;
      }
      if (t->state != Ticket::kDone) break;
    }
    if (ready == G) break;
    if (timeout_us == 0) return GC_PENDING;
    if (timeout_us > 0 && std::chrono::steady_clock::now() >= deadline) return GC_PENDING;
    poll_wait(b, &lk, began);
  }
  gc_status first = GC_OK;
  bool need_hi = false;
  static const uint64_t kZero[34] = {0};
  for (int64_t i = 0; i < G; ++i) {
    const Ticket* t = b->find(tickets[i]);
    if (!t) {  // retired while the lock was let go
      if (first == GC_OK) {
        first = GC_ERR_ARG;
        set_error("ticket " + std::to_string(i) + " is unknown or retired");
      }
      continue;
    }
    if (t->status != GC_OK && first == GC_OK) {
      first = t->status;
      set_error("the launch of ticket " + std::to_string(i) + " failed");
    }
    const uint64_t* x = t->out ? t->out->data() + 34 * (size_t)t->slot : kZero;
    for (int k = 0; k < 17; ++k) {
      global_out[17 * i + k] = x[2 * k];
      if (global_hi) global_hi[17 * i + k] = x[2 * k + 1];
      if (x[2 * k + 1]) need_hi = true;
    }
  }
  for (int64_t i = 0; i < G; ++i)
    if (b->find(tickets[i])) b->retire(tickets[i]);
  b->drop_retired();
  const bool rest = (b->flags & GC_BATCH_MANUAL) && idle(b);
  lk.unlock();
  if (rest) trim(b);
  if (first != GC_OK) return first;
  if (need_hi && !global_hi) {
    set_error("a global count exceeds 64 bits and global_hi is NULL");
    return GC_ERR_OVERFLOW;
  }
  return GC_OK;
} catch (...) {
  return no_memory();
}

gc_status gc_batch_destroy(gc_batch b) try {
  if (!b) return GC_OK;
  OutsideCapture relaxed;
  {
    std::lock_guard<std::mutex> lk(b->mu);
    b->stop = true;
  }
  b->cv.notify_all();
  if (b->dispatcher.joinable()) b->dispatcher.join();
  for (auto& s : b->streams) cudaStreamSynchronize(s);
  {
    std::lock_guard<std::mutex> lk(b->mu);
    retire_locked(b);
  }
  for (auto& sb : b->small) free_small_bufs(&sb);
  for (auto* f : b->forks) fork_release(f);
  for (Launch* L : b->spare) free_launch(L);
  reclaim_checks(b, true);
  for (Check& c : b->checks) {
    if (c.stream) {
      cudaStreamSynchronize(c.stream);
      cudaStreamDestroy(c.stream);
    }
    if (c.done) cudaEventDestroy(c.done);
    if (c.bad) cudaFreeHost(c.bad);
  }
  for (auto& s : b->streams) cudaStreamDestroy(s);
  delete b;
  return GC_OK;
} catch (...) {
  return no_memory();
}

}  // extern "C"
