// gc_run.cu -- the sequence of one count, shared by the whole-graph and the
// batched paths.
//
//   pass T  triangle step: |T| per edge, by lowest vertex         (Alg. 1)
//   pass C  4-cycles through every edge, degree-ordered wedges   (Alg. 4/6)
//   pass K  4-cliques and cross terms by lowest vertex           (Alg. 3/5)
//   finish  x10, per-edge columns, unrestricted sums             (Sec. 4.5)
//   derive  X_1..X_17                                            (Sec. 4.6)
//
// Everything is queued on the graph's stream, and on side streams forked from
// it and joined again, with no host synchronisation: the unit lists and their
// tier boundaries are fixed when the graph is prepared.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "gc_internal.h"

namespace gc {

namespace {
// Total bytes the pass-K global tier may hold at once.
constexpr size_t kKbufBudget = size_t(2) << 30;
// Graphs of fewer edges run pass C beside passes T and K.
constexpr int32_t kOverlapEdges = 1 << 22;
// Largest list of the edges of all H_a that pass T keeps for pass K.
constexpr long long kTListBudget = 24LL << 30;
// Largest per-CTA list of H_a edges in pass K (units with more edges rescan
// their out-lists instead): 2^19 entries, or the environment's GC_K_LIST_CAP
// (1 .. 2^19), read once per process.
long long k_list_cap() {
  static long long v = [] {
    const char* e = getenv("GC_K_LIST_CAP");
    long long x = e ? atoll(e) : (1LL << 19);
    return x < 1 ? 1LL : (x > (1LL << 19) ? (1LL << 19) : x);
  }();
  return v;
}
// Bound on the entries of pass T's edge lists from the environment's
// GC_T_LIST_CAP (>= 1; units past it scan again in pass K), read once per
// process; 0: not set.
long long t_list_cap_knob() {
  static long long v = [] {
    const char* e = getenv("GC_T_LIST_CAP");
    const long long x = e ? atoll(e) : 0;
    return e ? (x < 1 ? 1LL : x) : 0LL;
  }();
  return v;
}
}  // namespace

void scratch_free(Scratch* sc, cudaStream_t s) {
  for (void* p : {(void*)sc->zero, (void*)sc->tables, (void*)sc->kbuf, (void*)sc->hitbuf, (void*)sc->tlist,
                  (void*)sc->tl_off, (void*)sc->tl_cnt, (void*)sc->dsum, (void*)sc->vsum})
    if (p) cudaFreeAsync(p, s);
  *sc = Scratch();
}

gc_status scratch_init(Scratch* sc, int32_t m, int32_t table_n, int32_t kmax, const int32_t* tier_off, int32_t G,
                       int32_t dense_n, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
#define GS_TRY(call)                                \
  do {                                              \
    e = (call);                                     \
    if (e != cudaSuccess) return cuda_fail(e, "scratch alloc"); \
  } while (0)
  const size_t m1 = (size_t)(m > 0 ? m : 1);
  {
    size_t at = 0;
    auto take = [&](size_t bytes, size_t align = 16) {
      at = (at + align - 1) / align * align;
      const size_t o = at;
      at += bytes;
      return o;
    };
    const size_t misc = take(sizeof(int32_t) * 32), work = take(sizeof(unsigned long long) * kNumWork),
                 fill = take(sizeof(unsigned long long)),
                 csum = take(sizeof(unsigned long long) * 26 * (size_t)G),
                 x = take(sizeof(unsigned long long) * 34 * (size_t)G);
    sc->head_bytes = at;
    const size_t trio = take(sizeof(int32_t) * m1, 256), xc = take(sizeof(unsigned long long) * 2 * m1, 256),
                 P = take(sizeof(unsigned long long) * 2 * m1, 256),
                 x7d = take(sizeof(uint32_t) * (size_t)dense_n * (size_t)dense_n, 256);
    sc->zero_bytes = at;
    GS_TRY(pool_alloc(&sc->zero, at, s));
    sc->misc = reinterpret_cast<int32_t*>(sc->zero + misc);
    sc->work = reinterpret_cast<unsigned long long*>(sc->zero + work);
    sc->tl_fill = reinterpret_cast<unsigned long long*>(sc->zero + fill);
    sc->csum = reinterpret_cast<unsigned long long*>(sc->zero + csum);
    sc->x = reinterpret_cast<unsigned long long*>(sc->zero + x);
    sc->trio = reinterpret_cast<int32_t*>(sc->zero + trio);
    sc->xc = reinterpret_cast<unsigned long long*>(sc->zero + xc);
    sc->P = reinterpret_cast<unsigned long long*>(sc->zero + P);
    if (dense_n > 0) sc->x7d = reinterpret_cast<uint32_t*>(sc->zero + x7d);
  }
  if (table_n > kSmemTableMax) {
    sc->tables_n = (size_t)count_grid_size() * (size_t)table_n;
    GS_TRY(pool_alloc(&sc->tables, sizeof(uint32_t) * sc->tables_n, s));
    GS_TRY(cudaMemsetAsync(sc->tables, 0, sizeof(uint32_t) * sc->tables_n, s));
  }
  {  // passes T and K: each CTA records the edges of its current H_a (at most C(k, 2)); up to four CTAs per SM
    const int32_t ctas = 4 * (count_grid_size() / kCtasPerSm);
    int64_t at = 0;
    for (int t = 0; t < kTier32; ++t) {  // the warp tier keeps none
      const int32_t units = tier_off[t + 1] - tier_off[t];
      const int64_t k = t == kTierGlobal || kmax < kTierCap[t] ? kmax : kTierCap[t];
      const int64_t full = k * (k - 1) / 2;
      sc->hit_cap[t] = (int32_t)std::max<int64_t>(1, std::min<int64_t>(full, k_list_cap()));
      sc->hit_ctas[t] = std::min(units, ctas);
      sc->hit_off[t] = at;
      at += (int64_t)sc->hit_cap[t] * sc->hit_ctas[t];
    }
    GS_TRY(pool_alloc(&sc->hitbuf, sizeof(int2) * (size_t)std::max<int64_t>(1, at), s));
  }
  if (kmax > kTierCap[kTier1024]) {
    sc->kbuf_cap = kmax;
    sc->kbuf_stride = kbuf_bytes(kmax);
    size_t ctas = kKbufBudget / sc->kbuf_stride;
    const size_t sms = (size_t)(count_grid_size() / kCtasPerSm);
    if (ctas > sms) ctas = sms;
    if (ctas < 1) ctas = 1;
    sc->kbuf_ctas = (int32_t)ctas;
    GS_TRY(pool_alloc(&sc->kbuf, sc->kbuf_stride * ctas, s));
  }
#undef GS_TRY
  return GC_OK;
}

void scratch_guess_tlist(Scratch* sc, int64_t m) {
  const long long cap = kTListBudget / (long long)sizeof(int2);
  sc->tlist_want = 32 * m < cap ? 32 * m : cap;
}

static int32_t ku_total(const KUnits& ku) { return ku.tier_off[kNumTiers]; }

gc_status run_count(const DevGraph& g, const int32_t* units, int32_t n_units, const KUnits& ku,
                    uint64_t* per_edge, Scratch* sc, cudaStream_t s, ForkSet* fs, CountTimers* tm, bool per_edge_host,
                    uint64_t* induced, bool induced_host) {
  cudaError_t e = cudaSuccess;
  gc_status st = GC_OK;
#define GR_TRY(call, what)                  \
  do {                                      \
    e = (call);                             \
    if (e != cudaSuccess) return cuda_fail(e, what); \
  } while (0)
#define GR_BEGIN(i, t) \
  if (tm) GR_TRY(cudaEventRecord(tm->begin[i], t), "event")
#define GR_END(i, t) \
  if (tm) GR_TRY(cudaEventRecord(tm->end[i], t), "event")
  CountArgs a;
  a.units = units;
  a.n_units = n_units;
  a.kunits = ku.units;
  a.cunits = ku.cunits;
  a.n_cheavy = ku.n_cheavy;
  a.cjobs = ku.cjobs;
  a.n_cjobs = ku.n_cjobs;
  a.chash_w = ku.chash_w;
  a.n_chash = ku.n_chash;
  a.n_chash_big = ku.n_chash_big;
  a.n_chash_mid = ku.n_chash_mid;
  a.n_chash2_big = ku.n_chash2_big;
  a.n_chash2 = ku.n_chash2;
  a.hub_tab = hub_tab_words();
  for (int t = 0; t <= kNumTiers; ++t) a.ktier_off[t] = ku.tier_off[t];
  a.cursor = sc->misc;  // [0] pass C, [2 + tier] pass K, [8] pass C hubs, [9] pass C hashed, [10 + tier] pass T,
                        // [15] pass C packed-key hash, [7] pass C hashed small units,
                        // [16] pass C hashed middle units, [17] pass C packed-key hash, half tables
  a.status = sc->misc + 1;
  a.tables = g.table_n > kSmemTableMax ? sc->tables : nullptr;
  a.trio = sc->trio;
  a.P = sc->P;
  a.x7d = nullptr;
  a.xc = sc->xc;
  a.kbuf = sc->kbuf;
  a.kbuf_stride = sc->kbuf_stride;
  a.kbuf_ctas = sc->kbuf_ctas;
  a.kbuf_cap = sc->kbuf_cap;
  a.hitbuf = sc->hitbuf;
  for (int t = 0; t < kNumTiers; ++t) {
    a.hit_off[t] = sc->hit_off[t];
    a.hit_cap[t] = sc->hit_cap[t];
    a.hit_ctas[t] = sc->hit_ctas[t];
  }
  // Pass T keeps the edges of the H_a for pass K, in a list sized by the
  // triangles of the previous count of this scratch (or by a first guess);
  // units that do not fit scan their out-lists again in pass K.
  // Graphs of at most kSmemTableMax vertices may take the rows of common
  // neighbours instead of passes T and C (small_route); the per-edge induced
  // counts need pass T's degree sums.
  const bool rows = ku.rows && !(induced != nullptr && g.m > 0);
  if (!rows) {
    const int32_t nku = ku_total(ku);
    const long long want = sc->tlist_want;
    if (want > 0 && want * (long long)sizeof(int2) <= kTListBudget && nku > 0) {
      long long need = want + want / 16 + 1024;
      if (t_list_cap_knob() && need > t_list_cap_knob()) need = t_list_cap_knob();
      if (need > sc->tlist_cap) {
        if (sc->tlist) cudaFreeAsync(sc->tlist, s);
        sc->tlist = nullptr;
        sc->tlist_cap = 0;
        const long long cap = need;
        if (pool_alloc(&sc->tlist, sizeof(int2) * (size_t)cap, s) == cudaSuccess) sc->tlist_cap = cap;
        else cudaGetLastError();  // no list: pass K scans
      }
      if (nku > sc->tl_units) {
        for (void* p : {(void*)sc->tl_off, (void*)sc->tl_cnt})
          if (p) cudaFreeAsync(p, s);
        GR_TRY(pool_alloc(&sc->tl_off, sizeof(long long) * (size_t)nku, s), "alloc list index");
        GR_TRY(pool_alloc(&sc->tl_cnt, sizeof(int32_t) * (size_t)nku, s), "alloc list index");
        sc->tl_units = nku;
      }
    }
  }
  a.tlist = !rows && sc->tlist_cap > 0 ? sc->tlist : nullptr;
  a.tlist_cap = sc->tlist_cap;
  a.tlist_fill = sc->tl_fill;
  a.tl_off = sc->tl_off;
  a.tl_cnt = sc->tl_cnt;
  a.per_edge = per_edge;
  a.per_edge_host = per_edge != nullptr && per_edge_host;
  a.dsum = nullptr;
  const bool want_induced = induced != nullptr && g.m > 0;
  if (want_induced) {  // scratch of the per-edge induced counts, kept with the graph
    if (!sc->dsum) GR_TRY(pool_alloc(&sc->dsum, sizeof(unsigned long long) * (size_t)g.m, s), "alloc dsum");
    if (!sc->vsum)
      GR_TRY(pool_alloc(&sc->vsum, sizeof(unsigned long long) * 2 * (size_t)(g.n > 0 ? g.n : 1), s),
             "alloc vsum");
    GR_TRY(cudaMemsetAsync(sc->dsum, 0, sizeof(unsigned long long) * (size_t)g.m, s), "zero dsum");
    a.dsum = sc->dsum;
  }
  a.csum = sc->csum;
  a.work = sc->work;
  GR_TRY(cudaMemsetAsync(sc->zero, 0, sc->zero_bytes, s), "zero scratch");
  int launches = 0;
  // Pass C needs nothing of passes T and K. In graphs of fewer than
  // kOverlapEdges edges no pass fills the GPU for long (their kernels end in
  // tails of single units), so C runs beside T and K; above, the passes follow
  // each other, so that a pass's time says what it costs, with only the hub and
  // hash kernels of C side by side (16.8 -> 16.4 ms on Chung-Lu 10M edges; the
  // tiers of T and K gain nothing there). Chung-Lu, 500 009 edges: 1.06 -> 0.69
  // ms per count.
  const bool overlap = fs && g.m < kOverlapEdges;
  auto pass_c = [&](cudaStream_t t, Fork* fork) -> gc_status {
    const int32_t n_cunits = ku.n_cunits;  // pass C units: hubs, hashed units, the others
    if (n_cunits <= 0) return GC_OK;
    if (a.n_cheavy > 0) {
      if ((st = run_pass_c_heavy(g, a, t)) != GC_OK) return st;
      launches += 1;
    }
    if ((st = run_pass_c_hash2(g, a, fork, &launches)) != GC_OK) return st;
    if ((st = run_pass_c_hash(g, a, fork, &launches)) != GC_OK) return st;
    const int32_t n_hashed = a.n_cheavy + a.n_chash + a.n_chash2;
    if (n_cunits > n_hashed) {
      CountArgs al = a;  // the remaining units on the vertex-indexed tables
      al.units = a.cunits + n_hashed;
      al.n_units = n_cunits - n_hashed;
      if ((st = run_pass_c(g, al, t)) != GC_OK) return st;
      launches += 1;
    }
    return GC_OK;
  };
  auto pass_tk = [&](bool tri) -> gc_status {
    const Phase ph = tri ? kPhasePassT : kPhasePassK;
    GR_BEGIN(ph, s);
    Fork tiers(s, overlap ? fs : nullptr, 6, kForkStreams - 6);
    st = tri ? run_pass_t(g, a, &tiers, &launches) : run_pass_k(g, a, &tiers, &launches);
    if (st != GC_OK) return st;
    GR_TRY(tiers.join(), "join");
    GR_END(ph, s);
    return GC_OK;
  };
  if (rows) {
    GR_BEGIN(kPhasePassT, s);
    GR_END(kPhasePassT, s);
    // the dense kernels fill the GPU and want different shares of shared memory
    // and L1: side by side they take twice as long as one after the other
    const bool dense = g.bits != nullptr;
    if (dense) a.x7d = sc->x7d;
    // the rows stay on the count's stream, so that their kernel is the first on the
    // GPU: its largest vertex is the longest chain, and takes half as long again on an
    // SM that the cliques' kernels have filled before it (R-MAT scale 12: 240 us a
    // count, 270 to 295 when a side stream let them in first)
    Fork tiers(s, dense ? nullptr : fs, 6, kForkStreams - 6);
    if (!dense) GR_BEGIN(kPhasePassK, s);
    GR_BEGIN(kPhasePassC, s);
    if ((st = dense ? run_rows_dense(g, a, s) : run_rows(g, a, s)) != GC_OK) return st;
    launches += g.n > 0 ? 1 : 0;
    GR_END(kPhasePassC, s);
    if (dense) {
      GR_BEGIN(kPhasePassK, s);
      if ((st = run_cliques_dense(g, a, ku.kmax, s)) != GC_OK) return st;
      launches += ku_total(ku) > 0 ? 1 : 0;
    } else {
      if ((st = run_cliques_alone(g, a, &tiers, &launches)) != GC_OK) return st;
      GR_TRY(tiers.join(), "join");
    }
    GR_END(kPhasePassK, s);
  } else if (overlap) {
    // pass C on the set's first stream, its kernels forked from there
    Fork side(s, fs, 0, 1);
    const cudaStream_t t = side.next();
    GR_BEGIN(kPhasePassC, t);
    {
      Fork units(t, fs, 1, 5);
      if ((st = pass_c(t, &units)) != GC_OK) return st;
      GR_TRY(units.join(), "join");
    }
    GR_END(kPhasePassC, t);
    if ((st = pass_tk(true)) != GC_OK) return st;
    if ((st = pass_tk(false)) != GC_OK) return st;
    GR_TRY(side.join(), "join");
  } else {
    if ((st = pass_tk(true)) != GC_OK) return st;
    GR_BEGIN(kPhasePassC, s);
    {
      Fork units(s, fs, 1, 5);
      if ((st = pass_c(s, &units)) != GC_OK) return st;
      GR_TRY(units.join(), "join");
    }
    GR_END(kPhasePassC, s);
    if ((st = pass_tk(false)) != GC_OK) return st;
  }
  GR_BEGIN(kPhaseFinish, s);
  if ((st = run_finish(g, a, s)) != GC_OK) return st;
  launches += g.m > 0 ? 1 : 0;
  GR_END(kPhaseFinish, s);
  GR_BEGIN(kPhaseInduced, s);
  if (want_induced) {
    if ((st = run_induced(g, a, sc->vsum, induced, induced_host, s)) != GC_OK) return st;
    launches += g.n_long > 0 ? 3 : 2;
  }
  GR_END(kPhaseInduced, s);
  GR_BEGIN(kPhaseDerive, s);
  if ((st = run_derive(g, sc->csum, sc->x, a.status, s)) != GC_OK) return st;
  sc->launches = launches + 1;
  GR_END(kPhaseDerive, s);
  GR_BEGIN(kPhaseCopy, s);
#undef GR_BEGIN
#undef GR_END
#undef GR_TRY
  return GC_OK;
}

}  // namespace gc
