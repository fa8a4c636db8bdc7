// gc_api.cu -- C ABI of the plain whole-graph path (see include/gc.h).
//
// Host-side CSR validation (Problem 1's input: simple undirected graph) and
// the P1 relabelling, the graph handle with its device-resident data, and one
// count (the sequence of gc_run.cu: passes T, C, K, finish, derive) with the
// copies back.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "gc_internal.h"

namespace gc {

static thread_local std::string t_err;

void set_error(const std::string& msg) { t_err = msg; }

gc_status no_memory() noexcept {
  try {
    t_err = "host allocation failed";
  } catch (...) {
    t_err.clear();
  }
  return GC_ERR_NOMEM;
}

gc_status cuda_fail(cudaError_t e, const char* what) {
  set_error(std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")");
  if (e == cudaErrorMemoryAllocation) return GC_ERR_NOMEM;
  return GC_ERR_CUDA;
}

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pools[kMaxDevices] = {};
}  // namespace

cudaMemPool_t lib_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lk(g_pool_mu);
  if (g_pools[dev]) return g_pools[dev];
  cudaMemPoolProps props;
  std::memset(&props, 0, sizeof(props));
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  cudaMemPool_t pool = nullptr;
  if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) cudaGetLastError();
  unsigned long long keep = (unsigned long long)total_b / 4;
  if (const char* e = getenv("GC_POOL_KEEP_BYTES")) keep = strtoull(e, nullptr, 10);
  if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) cudaGetLastError();
  g_pools[dev] = pool;
  return pool;
}

namespace {
std::mutex g_fork_mu;
std::vector<ForkSet*> g_forks;          // idle sets, of any device
constexpr size_t kForksKept = 16;

void fork_destroy(ForkSet* f) {
  for (auto& t : f->stream)
    if (t) cudaStreamDestroy(t);
  for (cudaEvent_t e : f->done)
    if (e) cudaEventDestroy(e);
  if (f->start) cudaEventDestroy(f->start);
  delete f;
}
}  // namespace

ForkSet* fork_acquire(int dev, int priority) {
  {
    std::lock_guard<std::mutex> lk(g_fork_mu);
    for (size_t i = g_forks.size(); i-- > 0;)  // the last one given back
      if (g_forks[i]->device == dev && g_forks[i]->priority == priority) {
        ForkSet* f = g_forks[i];
        g_forks.erase(g_forks.begin() + (long)i);
        return f;
      }
  }
  ForkSet* f = new (std::nothrow) ForkSet();
  if (!f) {
    set_error("host allocation failed");
    return nullptr;
  }
  f->device = dev;
  f->priority = priority;
  const cudaError_t e = cudaEventCreateWithFlags(&f->start, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    cuda_fail(e, "side streams");
    fork_destroy(f);
    return nullptr;
  }
  return f;
}

bool on_part_of_gpu(cudaStream_t s) {
  typedef int (*Query)(cudaStream_t, void**);  // cuStreamGetGreenCtx
  static const Query query = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion("cuStreamGetGreenCtx", &f, 12040, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      f = nullptr;  // a driver without them
    }
    return reinterpret_cast<Query>(f);
  }();
  void* ctx = nullptr;
  return query && query(s, &ctx) == 0 && ctx != nullptr;
}

void fork_drain(ForkSet* f) {
  if (!f) return;
  for (auto& t : f->stream)
    if (t) cudaStreamSynchronize(t);
  cudaGetLastError();
}

void fork_release(ForkSet* f) {
  if (!f) return;
  {
    std::lock_guard<std::mutex> lk(g_fork_mu);
    try {
      if (g_forks.size() < kForksKept) {
        g_forks.push_back(f);
        return;
      }
    } catch (...) {  // no memory to keep it
    }
  }
  fork_destroy(f);
}

namespace {

// Timers of freed handles, kept for later ones (of any device: they are idle).
struct KeptTimers {
  CountTimers t;
  int device;
};
std::vector<KeptTimers> g_timers;  // under g_fork_mu
constexpr size_t kTimersKept = 16;

void timers_destroy(CountTimers* t) {
  for (cudaEvent_t e : t->begin)
    if (e) cudaEventDestroy(e);
  for (cudaEvent_t e : t->end)
    if (e) cudaEventDestroy(e);
  if (t->pinned) cudaFreeHost(t->pinned);
  *t = CountTimers();
}

cudaError_t timers_init(CountTimers* t, int dev) {
  {
    std::lock_guard<std::mutex> lk(g_fork_mu);
    for (size_t i = 0; i < g_timers.size(); ++i)
      if (g_timers[i].device == dev) {
        *t = g_timers[i].t;
        g_timers.erase(g_timers.begin() + (long)i);
        return cudaSuccess;
      }
  }
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < kNumPhases; ++k) {
    if (e == cudaSuccess) e = cudaEventCreate(&t->begin[k]);
    if (e == cudaSuccess) e = cudaEventCreate(&t->end[k]);
  }
  if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&t->pinned), kPinnedBytes);
  if (e != cudaSuccess) timers_destroy(t);
  return e;
}

void timers_release(CountTimers* t, int dev) {
  if (!t->pinned) return;  // never made
  {
    std::lock_guard<std::mutex> lk(g_fork_mu);
    try {
      if (g_timers.size() < kTimersKept) {
        g_timers.push_back({*t, dev});
        *t = CountTimers();
        return;
      }
    } catch (...) {  // no memory to keep them
    }
  }
  timers_destroy(t);
}

// Threads for a loop over `work` entries: one per 2^16, at most host_threads().
int threads_for(int64_t work) { return (int)std::max<int64_t>(1, std::min<int64_t>(host_threads(), work >> 16)); }

// Row ranges [b[t], b[t+1]) holding about equal numbers of entries.
std::vector<int32_t> nnz_chunks(int32_t n, const int32_t* rp, int nt) {
  std::vector<int32_t> b((size_t)nt + 1, n);
  b[0] = 0;
  const int64_t nnz = rp[n];
  for (int t = 1; t < nt; ++t) {
    const int32_t target = (int32_t)(nnz * t / nt);
    int32_t x = (int32_t)(std::upper_bound(rp, rp + n + 1, target) - rp) - 1;  // last row starting at or before
    if (x < b[t - 1]) x = b[t - 1];
    if (x > n) x = n;
    b[t] = x;
  }
  return b;
}

// For a graph that passed the linear checks (columns in range, rows
// ascending) and failed a symmetry check: the message naming the first entry
// (x, y) in row order whose reverse (y, x) is absent, found by a binary
// search in row y per entry (rows in chunks over the host threads). A walk's
// first mismatch need not be that entry -- an extra entry x0 in row y makes
// the next (x1, y) mismatch although (y, x1) exists -- so the failure path
// looks it up directly.
std::string first_without_reverse(int32_t n, const int32_t* rp, const int32_t* ci) {
  const int nt = threads_for(rp[n]);
  const std::vector<int32_t> b = nnz_chunks(n, rp, nt);
  std::vector<std::pair<int32_t, int32_t>> hit((size_t)nt, {-1, -1});
  host_run(nt, [&](int t) {
    for (int32_t x = b[t]; x < b[t + 1]; ++x)
      for (int32_t p = rp[x]; p < rp[x + 1]; ++p) {
        const int32_t y = ci[p];
        if (!std::binary_search(ci + rp[y], ci + rp[y + 1], x)) {
          hit[(size_t)t] = {x, y};
          return;
        }
      }
  });
  for (const auto& h : hit)
    if (h.first >= 0) return "edge (" + std::to_string(h.first) + "," + std::to_string(h.second) + ") has no reverse";
  return "asymmetric graph";  // not reached after a failed symmetry check
}

// First error of a multi-threaded check, by thread (thread order = row order).
struct Checks {
  std::vector<gc_status> st;
  std::vector<std::string> msg;
  explicit Checks(int nt) : st((size_t)nt, GC_OK), msg((size_t)nt) {}
  gc_status first() {
    for (size_t t = 0; t < st.size(); ++t)
      if (st[t] != GC_OK) {
        set_error(msg[t]);
        return st[t];
      }
    return GC_OK;
  }
};

}  // namespace

// Checks of Problem 1's input (a simple undirected graph), in two parts.
// Linear checks: row_ptr from 0 and non-decreasing, columns in range, rows
// strictly ascending (no duplicates), no self-loops -- one pass over the
// entries in threads over row ranges of equal entries.
// Whether a row passes every linear check (columns in [0, n), no self-loop,
// strictly ascending): no early exit and no branch in the loop, so that the
// compiler vectorises it; a failing row is examined again entry by entry.
static inline bool row_ok(const int32_t* r, int32_t len, int32_t x, int32_t n) {
  if (len <= 0) return true;
  uint32_t bad = ((uint32_t)r[0] >= (uint32_t)n) | (r[0] == x);
  for (int32_t k = 1; k < len; ++k)
    bad |= ((uint32_t)r[k] >= (uint32_t)n) | (r[k] == x) | (r[k] <= r[k - 1]);
  return bad == 0;
}

gc_status csr_linear_checks(int32_t n, const int32_t* rp, const int32_t* ci) {
  if (n < 0) { set_error("n < 0"); return GC_ERR_ARG; }
  if (rp[0] != 0) { set_error("row_ptr[0] != 0"); return GC_ERR_RANGE; }
  {  // row_ptr ascending: vertex chunks in parallel, the first decrease in row order
    const int ntv = threads_for(n);
    std::vector<int32_t> first((size_t)ntv, -1);
    host_run(ntv, [&](int t) {
      const int32_t x1 = (int32_t)((int64_t)n * (t + 1) / ntv);
      for (int32_t x = (int32_t)((int64_t)n * t / ntv); x < x1; ++x)
        if (rp[x + 1] < rp[x]) {
          first[(size_t)t] = x;
          return;
        }
    });
    for (int32_t x : first)
      if (x >= 0) {
        set_error("row_ptr decreases at row " + std::to_string(x));
        return GC_ERR_UNSORTED;
      }
  }
  if (rp[n] % 2 != 0) { set_error("row_ptr[n] is odd: the graph cannot be symmetric"); return GC_ERR_ASYMMETRIC; }
  const int64_t nnz = rp[n];
  const int nt = threads_for(nnz);
  const std::vector<int32_t> b = nnz_chunks(n, rp, nt);
  Checks c(nt);
  host_run(nt, [&](int t) {
    for (int32_t x = b[t]; x < b[t + 1]; ++x) {
      if (row_ok(ci + rp[x], rp[x + 1] - rp[x], x, n)) continue;
      for (int32_t p = rp[x]; p < rp[x + 1]; ++p) {  // the first failing entry of the first failing row
        const int32_t y = ci[p];
        if (y < 0 || y >= n) { c.st[t] = GC_ERR_RANGE; c.msg[t] = "column " + std::to_string(y) + " out of range in row " + std::to_string(x); return; }
        if (y == x) { c.st[t] = GC_ERR_SELF_LOOP; c.msg[t] = "self-loop at vertex " + std::to_string(x); return; }
        if (p > rp[x] && ci[p - 1] == y) { c.st[t] = GC_ERR_DUPLICATE; c.msg[t] = "duplicate neighbour " + std::to_string(y) + " in row " + std::to_string(x); return; }
        if (p > rp[x] && ci[p - 1] > y) { c.st[t] = GC_ERR_UNSORTED; c.msg[t] = "row " + std::to_string(x) + " not ascending"; return; }
      }
    }
  });
  return c.first();
}

// Symmetry (needs the linear checks passed): rows x are walked in order in
// chunks of about equal entries; the k-th row (in order) that names y must
// name it from the k-th entry of row y, so a per-chunk counter per y (started,
// on first use, at the number of entries of row y below the chunk's first
// row) gives the slot where x must stand in row y, and the entry there is
// compared with x. Every entry is checked against a slot of row y, so a
// missing reverse always fails, and a symmetric graph always passes. In graphs of
// fewer than 12 entries a vertex (whose counters every chunk clears for few
// entries each) the reverse of every upper entry (x, y), y > x, is searched
// instead: distinct upper entries find distinct lower ones, so the graph is
// symmetric if all are found and half of the entries are upper. All checks, 16
// cores, walk / search: 10^6 vertices and 6 entries each 15.7 / 9.8 ms, 10 each
// 24.2 / 17.3, 20 each 32.7 / 40.4; R-MAT scale 20, 30 each, 39.5 / 101. The
// message of a failure, naming the first entry in row order without a
// reverse, is returned in *msg (the calling thread sets it).
gc_status csr_symmetry(int32_t n, const int32_t* rp, const int32_t* ci, std::string* msg) {
  const int64_t nnz = rp[n];
  int nt = threads_for(nnz);
  // per-chunk counters: n ints per thread, at most 1 GiB in all
  const int64_t per = 4 * (int64_t)(n > 0 ? n : 1);
  nt = (int)std::max<int64_t>(1, std::min<int64_t>(nt, (int64_t(1) << 30) / per));
  const std::vector<int32_t> b = nnz_chunks(n, rp, nt);
  std::vector<gc_status> st((size_t)nt, GC_OK);
  if (nt > 1 && nnz < 12 * (int64_t)n) {
    std::vector<int64_t> upper((size_t)nt, 0);
    host_run(nt, [&](int t) {
      int64_t u = 0;
      for (int32_t x = b[t]; x < b[t + 1]; ++x) {
        const int32_t* e = ci + rp[x + 1];
        const int32_t* p = std::upper_bound(ci + rp[x], e, x);
        u += e - p;
        for (; p < e; ++p)
          if (!std::binary_search(ci + rp[*p], ci + rp[*p + 1], x)) {
            st[(size_t)t] = GC_ERR_ASYMMETRIC;
            return;
          }
      }
      upper[(size_t)t] = u;
    });
    int64_t total = 0;
    bool ok = true;
    for (int t = 0; t < nt; ++t) {
      total += upper[(size_t)t];
      ok &= st[(size_t)t] == GC_OK;
    }
    if (ok && 2 * total == nnz) return GC_OK;
    *msg = first_without_reverse(n, rp, ci);
    return GC_ERR_ASYMMETRIC;
  }
  host_run(nt, [&](int t) {
    std::vector<int32_t> fill((size_t)(n > 0 ? n : 1), -1);
    const int32_t x0 = b[t];
    for (int32_t x = x0; x < b[t + 1]; ++x)
      for (int32_t p = rp[x]; p < rp[x + 1]; ++p) {
        const int32_t y = ci[p];
        const int32_t yb = rp[y], ye = rp[y + 1];
        int32_t f = fill[y];
        if (f < 0) f = (int32_t)(std::lower_bound(ci + yb, ci + ye, x0) - (ci + yb));
        fill[y] = f + 1;
        const int32_t q = yb + f;
        if (q >= ye || ci[q] != x) {
          st[t] = GC_ERR_ASYMMETRIC;
          return;
        }
      }
  });
  for (int t = 0; t < nt; ++t)
    if (st[t] != GC_OK) {
      *msg = first_without_reverse(n, rp, ci);
      return st[t];
    }
  return GC_OK;
}

// The same checks, in the same order and with the same codes, for one small
// graph on the calling thread, with the caller's scratch for the symmetry
// walk (no allocation once the scratch has grown): what a bulk submission of
// many small graphs runs on each of its threads.
gc_status validate_csr_small(int32_t n, const int32_t* rp, const int32_t* ci, std::vector<int32_t>* fill) {
  if (n < 0) { set_error("n < 0"); return GC_ERR_ARG; }
  if (rp[0] != 0) { set_error("row_ptr[0] != 0"); return GC_ERR_RANGE; }
  for (int32_t x = 0; x < n; ++x)
    if (rp[x + 1] < rp[x]) {
      set_error("row_ptr decreases at row " + std::to_string(x));
      return GC_ERR_UNSORTED;
    }
  if (rp[n] % 2 != 0) { set_error("row_ptr[n] is odd: the graph cannot be symmetric"); return GC_ERR_ASYMMETRIC; }
  for (int32_t x = 0; x < n; ++x) {
    if (row_ok(ci + rp[x], rp[x + 1] - rp[x], x, n)) continue;
    for (int32_t p = rp[x]; p < rp[x + 1]; ++p) {
      const int32_t y = ci[p];
      if (y < 0 || y >= n) { set_error("column " + std::to_string(y) + " out of range in row " + std::to_string(x)); return GC_ERR_RANGE; }
      if (y == x) { set_error("self-loop at vertex " + std::to_string(x)); return GC_ERR_SELF_LOOP; }
      if (p > rp[x] && ci[p - 1] == y) { set_error("duplicate neighbour " + std::to_string(y) + " in row " + std::to_string(x)); return GC_ERR_DUPLICATE; }
      if (p > rp[x] && ci[p - 1] > y) { set_error("row " + std::to_string(x) + " not ascending"); return GC_ERR_UNSORTED; }
    }
  }
  // symmetry. The rows are sorted, so the entries of row y below y (its lower
  // part) must be, in order, the rows x < y that name y: each upper entry
  // (x, y), y > x, taken in row order, is matched with the next unmatched
  // entry of row y, which must be x; at the end every lower part must be
  // matched to its end. One random access per edge instead of one per entry;
  // a failure names the first entry in row order without a reverse, as for a
  // large graph.
  if ((int64_t)fill->size() < 2 * (int64_t)n) fill->resize(2 * (size_t)n);
  int32_t* f = fill->data();      // next unmatched entry of row y
  int32_t* lend = f + n;          // end of row x's lower part
  for (int32_t y = 0; y < n; ++y) f[y] = rp[y];
  bool sym = true;
  for (int32_t x = 0; x < n && sym; ++x) {
    int32_t p = rp[x];
    const int32_t e = rp[x + 1];
    while (p < e && ci[p] < x) ++p;
    lend[x] = p;
    for (; p < e; ++p) {
      const int32_t y = ci[p];
      const int32_t q = f[y]++;
      if (q >= rp[y + 1] || ci[q] != x) {
        sym = false;
        break;
      }
    }
  }
  for (int32_t y = 0; y < n && sym; ++y) sym = f[y] == lend[y];
  if (sym) return GC_OK;
  set_error(first_without_reverse(n, rp, ci));
  return GC_ERR_ASYMMETRIC;
}

gc_status validate_csr(int32_t n, const int32_t* rp, const int32_t* ci) {
  if (n >= 0 && rp[n] >= 0 && rp[n] < (1 << 17)) {
    std::vector<int32_t> fill;
    return validate_csr_small(n, rp, ci, &fill);
  }
  gc_status st = csr_linear_checks(n, rp, ci);
  if (st != GC_OK) return st;
  std::string msg;
  st = csr_symmetry(n, rp, ci, &msg);
  if (st != GC_OK) set_error(msg);
  return st;
}

RelabelPlan plan_relabel(int32_t n, const int32_t* rp, int max_threads) {
  RelabelPlan R;
  R.perm.resize((size_t)n);
  R.newid.resize((size_t)n);
  R.rp.resize((size_t)n + 1);
  R.rp[0] = 0;
  if (n == 0) return R;
  // vertex chunks, one per thread (fewer threads when the per-thread degree
  // histograms would pass 2^24 counters)
  int nt = std::min(threads_for(n), max_threads);
  std::vector<int32_t> dmx((size_t)nt, 0);
  auto chunk = [&](int t, int T) { return (int32_t)((int64_t)n * t / T); };
  host_run(nt, [&](int t) {
    int32_t d = 0;
    for (int32_t x = chunk(t, nt); x < chunk(t + 1, nt); ++x) d = std::max(d, rp[x + 1] - rp[x]);
    dmx[(size_t)t] = d;
  });
  const int32_t dmax = *std::max_element(dmx.begin(), dmx.end());
  const size_t D = (size_t)dmax + 1;
  const int nt0 = nt;
  while (nt > 1 && (size_t)nt * D > ((size_t)1 << 24)) nt >>= 1;
  if (nt != nt0) dmx.assign((size_t)nt, 0);
  // cnt[t][d]: vertices of degree d in chunk t, then the first rank each
  // chunk gives its degree-d vertices: ranks ascend by degree, then by chunk,
  // then by id within the chunk -- the (degree, id) order
  std::vector<int32_t> cnt((size_t)nt * D, 0);
  host_run(nt, [&](int t) {
    int32_t* c = cnt.data() + (size_t)t * D;
    for (int32_t x = chunk(t, nt); x < chunk(t + 1, nt); ++x) c[rp[x + 1] - rp[x]]++;
  });
  std::vector<int32_t> base(D + 1);  // first rank of degree d
  std::vector<int64_t> S(D + 1);     // first internal slot of degree d
  {
    int32_t r = 0;
    int64_t sl = 0;
    for (size_t d = 0; d < D; ++d) {
      base[d] = r;
      S[d] = sl;
      int32_t tot = 0;
      for (int t = 0; t < nt; ++t) {
        int32_t& c = cnt[(size_t)t * D + d];
        const int32_t k = c;
        c = r + tot;  // chunk t's first rank of degree d
        tot += k;
      }
      r += tot;
      sl += (int64_t)tot * (int64_t)d;
    }
    base[D] = r;
    S[D] = sl;
  }
  for (int k = 0; k < kOBounds; ++k) R.obound[k] = base[std::min<size_t>((size_t)kOBoundDeg[k], D)];
  host_run(nt, [&](int t) {
    int32_t* c = cnt.data() + (size_t)t * D;
    for (int32_t x = chunk(t, nt); x < chunk(t + 1, nt); ++x) {
      const int32_t i = c[rp[x + 1] - rp[x]]++;
      R.perm[(size_t)i] = x;
      R.newid[(size_t)x] = i;
    }
  });
  // internal row pointers: every row of a degree bucket has that degree
  host_run(nt, [&](int t) {
    for (int32_t i = chunk(t, nt); i < chunk(t + 1, nt); ++i) {
      const int32_t x = R.perm[(size_t)i];
      const int32_t d = rp[x + 1] - rp[x];
      R.rp[(size_t)i + 1] = (int32_t)(S[(size_t)d] + (int64_t)(i + 1 - base[(size_t)d]) * d);
    }
  });
  // rows of 33..4096 entries and longer ones: the last ranks, in two runs
  const int32_t m0 = base[std::min<size_t>(33, D)], l0 = base[std::min<size_t>(4097, D)];
  R.mid.resize((size_t)(l0 - m0));
  for (int32_t i = m0; i < l0; ++i) R.mid[(size_t)(i - m0)] = i;
  for (int32_t i = l0; i < n; ++i) {
    const int32_t d = R.rp[(size_t)i + 1] - R.rp[(size_t)i];
    int64_t P = 4096;
    while (P < d) P <<= 1;
    R.longr.push_back(i);
    R.long_off.push_back(R.tmp_len);
    R.tmp_len += P;
  }
  return R;
}

}  // namespace gc

using namespace gc;

struct gc_graph_s {
  int32_t n = 0;
  int32_t m = 0;
  cudaStream_t stream = nullptr;
  int32_t* d_rp = nullptr;
  int32_t* d_ci = nullptr;
  PrepBuffers prep;
  // single-graph descriptors (G = 1)
  int32_t* d_gbase = nullptr;  // [1] 0
  int32_t* d_gn = nullptr;     // [1] n
  int64_t* d_gm = nullptr;     // [1] m
  // counting scratch
  Scratch sc;
  uint64_t* d_pe_tmp = nullptr;          // device staging for a host per-edge buffer
  uint64_t* d_ind_tmp = nullptr;         // device staging for a host per-edge induced buffer
  int32_t n_long = 0;                    // rows of more than 4096 entries
  int priority = 0;                      // of the stream
  bool part = false;                     // it is on a part of the GPU
  int device = 0;
  CountTimers timers;                    // events of the last count, and the pinned results
  bool counted = false;
  uint64_t csum_lo[13] = {0}, csum_hi[13] = {0};
  uint64_t work[kNumWork] = {0};
};

extern "C" {

const char* gc_last_error(void) { return t_err.c_str(); }

gc_status gc_validate_csr(int32_t n, const int32_t* row_ptr, const int32_t* col_idx) try {
  if (n < 0 || !row_ptr || (!col_idx && n > 0 && row_ptr[n] > 0)) {
    set_error("bad arguments to gc_validate_csr");
    return GC_ERR_ARG;
  }
  if (row_ptr[n] >= 0 && row_ptr[n] < (1 << 20)) {
    // the single-threaded checks each graph of a bulk submission gets
    std::vector<int32_t> fill;
    return validate_csr_small(n, row_ptr, col_idx, &fill);
  }
  return validate_csr(n, row_ptr, col_idx);
} catch (...) {
  return no_memory();
}

static void graph_release(gc_graph g) {
  if (!g) return;
  // stream-ordered frees into the library pool (after the graph's queued
  // work), then one synchronisation
  const cudaStream_t s = g->stream;
  for (void* p : {(void*)g->d_rp, (void*)g->d_ci, (void*)g->d_gbase, (void*)g->d_pe_tmp,
                  (void*)g->d_ind_tmp})
    if (p) cudaFreeAsync(p, s);
  free_prep(&g->prep, s);
  scratch_free(&g->sc, s);
  cudaStreamSynchronize(s);
  timers_release(&g->timers, g->device);
  delete g;
}

gc_status gc_graph_upload(int32_t n, const int32_t* row_ptr, const int32_t* col_idx, uint32_t flags,
                          void* stream, gc_graph* out) try {
  if (!out) { set_error("out is NULL"); return GC_ERR_ARG; }
  *out = nullptr;
  if (n < 0 || !row_ptr || (!col_idx && n > 0 && row_ptr[n] > 0)) {
    set_error("bad arguments to gc_graph_upload");
    return GC_ERR_ARG;
  }
  if (flags & ~GC_NO_VALIDATE) { set_error("unknown flags"); return GC_ERR_ARG; }
  const bool validate = !(flags & GC_NO_VALIDATE);
  if (validate) {
    const gc_status st0 = csr_linear_checks(n, row_ptr, col_idx);
    if (st0 != GC_OK) return st0;
  }
  const int64_t nnz = row_ptr[n];
  if (nnz < 0 || nnz % 2) { set_error("row_ptr[n] must be even and >= 0"); return GC_ERR_ARG; }
  // Symmetry is checked on the device, where the preparation finds the
  // reverse of every slot: the device steps are safe on an asymmetric input
  // (columns in range, rows sorted), and nothing is counted before the check
  // has passed. If a device step fails, the host checks symmetry instead, so
  // that an invalid input is reported as such (also where there is no GPU).
  gc_graph g = new (std::nothrow) gc_graph_s();
  if (!g) { set_error("host allocation failed"); return GC_ERR_NOMEM; }
  g->n = n;
  g->m = (int32_t)(nnz / 2);
  g->stream = (cudaStream_t)stream;
  if (cudaGetDevice(&g->device) != cudaSuccess) cudaGetLastError();  // the first device step reports it
  cudaStream_t s = g->stream;
  cudaError_t e;
  gc_status st = GC_OK;
  RelabelPlan R;
  int32_t *d_eid = nullptr, *d_perm = nullptr, *d_newid = nullptr, *d_rp0 = nullptr, *d_ci0 = nullptr;
  int32_t* d_lists = nullptr;
  long long* d_tmp = nullptr;
  int64_t* d_loff = nullptr;
  auto drop_temps = [&] {
    for (void* p : {(void*)d_newid, (void*)d_rp0, (void*)d_ci0, (void*)d_lists, (void*)d_tmp, (void*)d_loff})
      if (p) cudaFreeAsync(p, s);
    d_newid = d_rp0 = d_ci0 = d_lists = nullptr;
    d_tmp = nullptr;
    d_loff = nullptr;
  };
  // On a failure the symmetry check is awaited first: an invalid input is
  // reported as such even when a device step failed too (a machine without a
  // GPU still gets the validation codes).
  auto fail = [&](gc_status code) -> gc_status {
    const std::string err = gc_last_error();
    drop_temps();
    if (d_eid) cudaFreeAsync(d_eid, s);
    if (d_perm) cudaFreeAsync(d_perm, s);
    graph_release(g);
    if (validate) {
      std::string msg;
      const gc_status sym_st = csr_symmetry(n, row_ptr, col_idx, &msg);
      if (sym_st != GC_OK) {
        set_error(msg);
        return sym_st;
      }
    }
    set_error(err);
    return code;
  };
#define GC_CHECK(call, what)            \
  do {                                  \
    e = (call);                         \
    if (e != cudaSuccess) return fail(cuda_fail(e, what)); \
  } while (0)
  try {
    R = plan_relabel(n, row_ptr, host_threads());
  } catch (...) {
    set_error("host allocation failed");
    return fail(GC_ERR_NOMEM);
  }
  g->n_long = (int32_t)R.longr.size();
  const size_t nnz1 = (size_t)(nnz > 0 ? nnz : 1), n1 = (size_t)(n > 0 ? n : 1);
  const size_t n_lists = R.mid.size() + R.longr.size();
  GC_CHECK(pool_alloc(&g->d_rp, sizeof(int32_t) * ((size_t)n + 1), s), "alloc row_ptr");
  GC_CHECK(pool_alloc(&g->d_ci, sizeof(int32_t) * nnz1, s), "alloc col_idx");
  GC_CHECK(pool_alloc(&d_eid, sizeof(int32_t) * nnz1, s), "alloc eid");
  GC_CHECK(pool_alloc(&d_perm, sizeof(int32_t) * n1, s), "alloc perm");
  GC_CHECK(pool_alloc(&d_newid, sizeof(int32_t) * n1, s), "alloc newid");
  GC_CHECK(pool_alloc(&d_rp0, sizeof(int32_t) * ((size_t)n + 1), s), "alloc caller row_ptr");
  GC_CHECK(pool_alloc(&d_ci0, sizeof(int32_t) * nnz1, s), "alloc caller col_idx");
  GC_CHECK(pool_alloc(&d_lists, sizeof(int32_t) * (n_lists > 0 ? n_lists : 1), s), "alloc row lists");
  GC_CHECK(pool_alloc(&d_loff, sizeof(int64_t) * (R.long_off.size() > 0 ? R.long_off.size() : 1), s),
           "alloc row lists");
  GC_CHECK(pool_alloc(&d_tmp, sizeof(long long) * (size_t)(R.tmp_len > 0 ? R.tmp_len : 1), s), "alloc sort buffer");
  GC_CHECK(cudaMemcpyAsync(d_rp0, row_ptr, sizeof(int32_t) * ((size_t)n + 1), cudaMemcpyHostToDevice, s),
           "copy row_ptr");
  if (nnz > 0)
    GC_CHECK(cudaMemcpyAsync(d_ci0, col_idx, sizeof(int32_t) * (size_t)nnz, cudaMemcpyHostToDevice, s), "copy col_idx");
  GC_CHECK(cudaMemcpyAsync(g->d_rp, R.rp.data(), sizeof(int32_t) * ((size_t)n + 1), cudaMemcpyHostToDevice, s),
           "copy internal row_ptr");
  if (n > 0) {
    GC_CHECK(cudaMemcpyAsync(d_perm, R.perm.data(), sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, s), "copy perm");
    GC_CHECK(cudaMemcpyAsync(d_newid, R.newid.data(), sizeof(int32_t) * (size_t)n, cudaMemcpyHostToDevice, s),
             "copy ranks");
  }
  if (!R.mid.empty())
    GC_CHECK(cudaMemcpyAsync(d_lists, R.mid.data(), sizeof(int32_t) * R.mid.size(), cudaMemcpyHostToDevice, s),
             "copy row lists");
  if (!R.longr.empty()) {
    GC_CHECK(cudaMemcpyAsync(d_lists + R.mid.size(), R.longr.data(), sizeof(int32_t) * R.longr.size(),
                             cudaMemcpyHostToDevice, s), "copy row lists");
    GC_CHECK(cudaMemcpyAsync(d_loff, R.long_off.data(), sizeof(int64_t) * R.long_off.size(), cudaMemcpyHostToDevice, s),
             "copy row lists");
  }
  st = relabel_on_device(n, g->m, d_rp0, d_ci0, d_perm, d_newid, g->d_rp, g->d_ci, d_eid, nullptr, nullptr, d_lists,
                         (int32_t)R.mid.size(), d_lists + R.mid.size(), d_loff, (int32_t)R.longr.size(), d_tmp, s);
  drop_temps();
  if (st != GC_OK) return fail(st);
  const int32_t zero = 0;
  const RankInfo rank = {R.rp.data(), 1, &zero, &n, R.obound, nullptr, nullptr};
  st = prepare_graph(n, g->m, g->d_rp, g->d_ci, d_eid, d_perm, rank, &g->prep, s);
  d_eid = nullptr;  // owned by the preparation buffers from here on
  if (st != GC_OK) return fail(st);
  cudaFreeAsync(d_perm, s);
  d_perm = nullptr;
  if (validate) {
    int32_t bad = -1;
    if ((st = first_unreversed_slot(nnz, g->prep.rev, &bad, s)) != GC_OK) return fail(st);
    if (bad >= 0) {  // name the edge in the caller's labels
      int32_t y = 0;
      GC_CHECK(cudaMemcpy(&y, g->d_ci + bad, sizeof(int32_t), cudaMemcpyDeviceToHost), "copy slot");
      const int32_t x = (int32_t)(std::upper_bound(R.rp.data(), R.rp.data() + n + 1, bad) - R.rp.data()) - 1;
      set_error("edge (" + std::to_string(R.perm[x]) + "," + std::to_string(R.perm[y]) + ") has no reverse");
      graph_release(g);
      return GC_ERR_ASYMMETRIC;
    }
  }
  cudaStreamSynchronize(s);  // the host arrays of the plan are released on return
  // single-graph descriptor block: gbase | gn | gm (gm 8-byte aligned)
  GC_CHECK(pool_alloc(&g->d_gbase, 32, s), "alloc descriptors");
  {
    int32_t hb[4] = {0, n, 0, 0};
    int64_t hm = g->m;
    GC_CHECK(cudaMemcpyAsync(g->d_gbase, hb, 16, cudaMemcpyHostToDevice, s), "copy descriptors");
    GC_CHECK(cudaMemcpyAsync(reinterpret_cast<char*>(g->d_gbase) + 16, &hm, 8, cudaMemcpyHostToDevice, s),
             "copy descriptors");
    g->d_gn = g->d_gbase + 1;
    g->d_gm = reinterpret_cast<int64_t*>(reinterpret_cast<char*>(g->d_gbase) + 16);
  }
  {
    gc_status st2 = GC_OK;
    if (g->prep.route == kRouteDense) st2 = build_bits(n, g->d_rp, g->d_ci, &g->prep, s);
    if (st2 == GC_OK)
      st2 = scratch_init(&g->sc, g->m, needs_tables(g->prep) ? n : 0, g->prep.kmax, g->prep.ktier_off, 1,
                         g->prep.bits ? n : 0, s);
    if (st2 != GC_OK) return fail(st2);
    scratch_guess_tlist(&g->sc, g->m);
  }
  GC_CHECK(timers_init(&g->timers, g->device), "events");
  if (cudaStreamGetPriority(s, &g->priority) != cudaSuccess) cudaGetLastError();
  g->part = on_part_of_gpu(s);
  GC_CHECK(cudaStreamSynchronize(s), "sync upload");
#undef GC_CHECK
  *out = g;
  return GC_OK;
} catch (...) {
  return no_memory();
}

gc_status gc_graph_info(gc_graph g, int64_t* n, int64_t* m) {
  if (!g) { set_error("graph is NULL"); return GC_ERR_ARG; }
  if (n) *n = g->n;
  if (m) *m = g->m;
  return GC_OK;
}

gc_status gc_graph_edges(gc_graph g, int32_t* uv) try {
  if (!g || !uv) { set_error("NULL argument"); return GC_ERR_ARG; }
  if (g->m == 0) return GC_OK;
  cudaError_t e = cudaMemcpyAsync(uv, g->prep.uv, sizeof(int32_t) * 2 * (size_t)g->m,
                                  cudaMemcpyDeviceToHost, g->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(g->stream);
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "copy edges");
} catch (...) {
  return no_memory();
}

// The address by which the device writes the per-edge rows at p: p itself
// for device or managed memory, the mapped address for pinned host memory
// (the finish kernel then writes the rows over the host link, with no staging
// buffer and no copy; *host = true), nullptr for pageable host memory.
static uint64_t* device_view(uint64_t* p, bool* host) {
  *host = false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) return p;
  if (a.type == cudaMemoryTypeHost && a.devicePointer) {
    *host = true;
    return static_cast<uint64_t*>(a.devicePointer);
  }
  return nullptr;
}

// The count behind gc_count_edge_graphlets and gc_count_edge_induced.
static gc_status count_graph(gc_graph g, uint64_t* per_edge_out, uint64_t* induced_out, uint64_t* global_out,
                             uint64_t* global_hi) {
  if (!g || !global_out) { set_error("NULL argument"); return GC_ERR_ARG; }
  cudaStream_t s = g->stream;
  cudaError_t e;
  gc_status st;
  // the side streams are the current device's, and so would their kernels be
  int dev = -1;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev != g->device) {
    set_error("the graph is on device " + std::to_string(g->device) + ", the current device is " + std::to_string(dev));
    return GC_ERR_CUDA;
  }
#define GC_CHECK(call, what)                  \
  do {                                        \
    e = (call);                               \
    if (e != cudaSuccess) return cuda_fail(e, what); \
  } while (0)
  uint64_t* pe_dev = nullptr;
  const bool want_pe = per_edge_out != nullptr && g->m > 0;
  bool staged = false, pe_host = false;
  if (want_pe) {
    if ((pe_dev = device_view(per_edge_out, &pe_host)) == nullptr) {
      staged = true;
      if (!g->d_pe_tmp)
        GC_CHECK(pool_alloc(&g->d_pe_tmp, sizeof(uint64_t) * 13 * (size_t)g->m, g->stream), "alloc per-edge staging");
      pe_dev = g->d_pe_tmp;
    }
  }
  uint64_t* ind_dev = nullptr;
  const bool want_ind = induced_out != nullptr && g->m > 0;
  bool ind_staged = false, ind_host = false;
  if (want_ind) {
    if ((ind_dev = device_view(induced_out, &ind_host)) == nullptr) {
      ind_staged = true;
      if (!g->d_ind_tmp)
        GC_CHECK(pool_alloc(&g->d_ind_tmp, sizeof(uint64_t) * GC_INDUCED_COLS * (size_t)g->m, g->stream),
                 "alloc induced staging");
      ind_dev = g->d_ind_tmp;
    }
  }
  DevGraph dg;
  dg.n = g->n;
  dg.m = g->m;
  dg.rp = g->d_rp;
  dg.ci = g->d_ci;
  dg.deg = g->prep.deg;
  dg.eid = g->prep.eid;
  dg.out_ptr = g->prep.out_ptr;
  dg.out_idx = g->prep.out_idx;
  dg.ocsr = g->prep.ocsr;
  dg.e2o = g->prep.e2o;
  dg.rev = g->prep.rev;
  dg.G = 1;
  dg.vgid = nullptr;
  dg.gbase = g->d_gbase;
  dg.gn = g->d_gn;
  dg.gm = g->d_gm;
  dg.table_n = g->n;
  dg.bits = g->prep.bits;
  dg.bits_t = g->prep.bits_t;
  dg.hgeom = g->prep.hgeom;
  dg.hseg = g->prep.hseg;
  dg.hpos = g->prep.hpos;
  dg.n_long = g->n_long;
  KUnits ku;
  ku.kmax = g->prep.kmax;
  ku.units = g->prep.kunits;
  ku.cunits = g->prep.cunits;
  ku.n_cheavy = g->prep.n_cheavy;
  ku.cjobs = g->prep.cjobs;
  ku.n_cjobs = g->prep.n_cjobs;
  ku.chash_w = g->prep.chash_w;
  ku.n_chash = g->prep.n_chash;
  ku.n_chash2 = g->prep.n_chash2;
  ku.n_chash_big = g->prep.n_chash_big;
  ku.n_chash_mid = g->prep.n_chash_mid;
  ku.n_chash2_big = g->prep.n_chash2_big;
  ku.n_cunits = g->prep.n_cunits;
  ku.rows = g->prep.route != kRoutePasses;
  for (int t = 0; t <= kNumTiers; ++t) ku.tier_off[t] = g->prep.ktier_off[t];
  struct Lent {  // the side streams of this count, idle again when it ends
    ForkSet* f;
    bool joined = false;
    ~Lent() {
      if (!joined) fork_drain(f);
      fork_release(f);
    }
  } lent = {nullptr};
  // what the default streams stand for is the current context's to say
  const bool part = (uintptr_t)s <= (uintptr_t)cudaStreamPerThread ? on_part_of_gpu(s) : g->part;
  if (!part && !(lent.f = fork_acquire(dev, g->priority))) return GC_ERR_CUDA;
  if ((st = run_count(dg, g->prep.units, g->prep.n_units, ku, pe_dev, &g->sc, s, lent.f, &g->timers, pe_host, ind_dev,
                      ind_host)) != GC_OK)
    return st;
  // the results' head of the scratch in one copy: status, work, sums, X
  if (g->sc.head_bytes > kPinnedBytes) { set_error("internal: results do not fit"); return GC_ERR_CUDA; }
  GC_CHECK(cudaMemcpyAsync(g->timers.pinned, g->sc.zero, g->sc.head_bytes, cudaMemcpyDeviceToHost, s), "copy results");
  if (staged)
    GC_CHECK(cudaMemcpyAsync(per_edge_out, pe_dev, sizeof(uint64_t) * 13 * (size_t)g->m, cudaMemcpyDeviceToHost, s),
             "copy per-edge");
  if (ind_staged)
    GC_CHECK(cudaMemcpyAsync(induced_out, ind_dev, sizeof(uint64_t) * GC_INDUCED_COLS * (size_t)g->m,
                             cudaMemcpyDeviceToHost, s),
             "copy induced");
  GC_CHECK(cudaEventRecord(g->timers.end[kPhaseCopy], s), "event");
  GC_CHECK(cudaStreamSynchronize(s), "sync count");
  lent.joined = true;
  auto host_of = [&](const void* d) { return g->timers.pinned + (static_cast<const unsigned char*>(d) - g->sc.zero); };
  const int32_t hstatus = reinterpret_cast<const int32_t*>(host_of(g->sc.misc))[1];
  std::memcpy(g->work, host_of(g->sc.work), sizeof(g->work));
  const uint64_t* hx = reinterpret_cast<const uint64_t*>(host_of(g->sc.x));
  const uint64_t* hc = reinterpret_cast<const uint64_t*>(host_of(g->sc.csum));
  g->sc.tlist_want = (long long)g->work[kWorkTTriangles];  // the next count keeps pass T's edge lists
#undef GC_CHECK
  if (hstatus & kSpillOverflow) {
    set_error("internal: a unit outgrew its tier or hash (only for input that skipped validation)");
    return GC_ERR_CUDA;
  }
  if (hstatus & kInexact) {
    set_error("internal: a global relation had a non-zero remainder");
    return GC_ERR_CUDA;
  }
  bool need_hi = false;
  for (int i = 0; i < 17; ++i) {
    global_out[i] = hx[2 * i];
    if (global_hi) global_hi[i] = hx[2 * i + 1];
    if (hx[2 * i + 1]) need_hi = true;
  }
  for (int k = 0; k < 13; ++k) {
    g->csum_lo[k] = hc[2 * k];
    g->csum_hi[k] = hc[2 * k + 1];
  }
  g->counted = true;
  if (need_hi && !global_hi) {
    set_error("a global count exceeds 64 bits and global_hi is NULL");
    return GC_ERR_OVERFLOW;
  }
  return GC_OK;
}

gc_status gc_count_edge_graphlets(gc_graph g, uint64_t* per_edge_out, uint64_t* global_out,
                                  uint64_t* global_hi) try {
  return count_graph(g, per_edge_out, nullptr, global_out, global_hi);
} catch (...) {
  return no_memory();
}

gc_status gc_count_edge_induced(gc_graph g, uint64_t* induced_out, uint64_t* per_edge_out, uint64_t* global_out,
                                uint64_t* global_hi) try {
  if (!induced_out && g && g->m > 0) { set_error("induced_out is NULL"); return GC_ERR_ARG; }
  return count_graph(g, per_edge_out, induced_out, global_out, global_hi);
} catch (...) {
  return no_memory();
}

gc_status gc_graph_csums(gc_graph g, uint64_t* lo, uint64_t* hi) {
  if (!g || !lo) { set_error("NULL argument"); return GC_ERR_ARG; }
  if (!g->counted) { set_error("graph not counted yet"); return GC_ERR_ARG; }
  for (int k = 0; k < 13; ++k) {
    lo[k] = g->csum_lo[k];
    if (hi) hi[k] = g->csum_hi[k];
  }
  return GC_OK;
}

gc_status gc_graph_work_counts(gc_graph g, uint64_t* out) {
  if (!g || !out) { set_error("NULL argument"); return GC_ERR_ARG; }
  if (!g->counted) { set_error("graph not counted yet"); return GC_ERR_ARG; }
  static_assert(kNumWork == GC_NUM_WORK, "work counter count");
  for (int i = 0; i < kNumWork; ++i) out[i] = g->work[i];
  out[kWorkLaunches] = (uint64_t)g->sc.launches;
  return GC_OK;
}

int gc_phase_count(void) { return kNumPhases; }

const char* gc_phase_name(int i) {
  static const char* names[kNumPhases] = {"pass_t_triangles", "pass_c_cycles", "pass_k_cliques",
                                          "finish_columns", "induced_columns", "derive", "copy_out"};
  return (i >= 0 && i < kNumPhases) ? names[i] : "";
}

gc_status gc_graph_phase_ms(gc_graph g, double* ms) {
  if (!g || !ms) { set_error("NULL argument"); return GC_ERR_ARG; }
  if (!g->counted) { set_error("graph not counted yet"); return GC_ERR_ARG; }
  for (int i = 0; i < kNumPhases; ++i) {
    float f = 0.f;
    cudaError_t e = cudaEventElapsedTime(&f, g->timers.begin[i], g->timers.end[i]);
    if (e != cudaSuccess) return cuda_fail(e, "event elapsed");
    ms[i] = f;
  }
  return GC_OK;
}

gc_status gc_graph_free(gc_graph g) {
  graph_release(g);
  return GC_OK;
}

// The idle side streams and timers of the current device, given back.
static void fork_trim() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  std::lock_guard<std::mutex> lk(g_fork_mu);
  for (size_t i = g_forks.size(); i-- > 0;)
    if (g_forks[i]->device == dev) {
      fork_destroy(g_forks[i]);
      g_forks.erase(g_forks.begin() + (long)i);
    }
  for (size_t i = g_timers.size(); i-- > 0;)
    if (g_timers[i].device == dev) {
      timers_destroy(&g_timers[i].t);
      g_timers.erase(g_timers.begin() + (long)i);
    }
}

gc_status gc_release_cached_memory(void) try {
  cudaMemPool_t pool = lib_pool();
  if (!pool) {
    set_error("gc_release_cached_memory: no CUDA device or pool");
    return GC_ERR_CUDA;
  }
  cudaError_t e = cudaDeviceSynchronize();  // every stream-ordered free has reached the pool
  if (e == cudaSuccess) e = cudaMemPoolTrimTo(pool, 0);
  fork_trim();
  return e == cudaSuccess ? GC_OK : cuda_fail(e, "gc_release_cached_memory");
} catch (...) {
  return no_memory();
}

}  // extern "C"
