// gc_deal.h -- work of a warp dealt to its lanes: runs of different lengths end to
// end, and the rows of consecutive CSR slots.
#pragma once

#include <stdint.h>

namespace gc {

// Runs of 32 lanes laid end to end: lane ranks of the non-empty runs, for
// the owner lookup of deal_owner (call with the whole warp).
struct Deal {
  int32_t excl, total;
  unsigned nz;
};
__device__ __forceinline__ Deal deal_setup(int32_t L, int32_t* comp, int lane) {
  Deal d;
  int32_t incl = L;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  d.excl = incl - L;
  d.total = __shfl_sync(0xffffffffu, incl, 31);
  d.nz = __ballot_sync(0xffffffffu, L > 0);
  if (L > 0) comp[__popc(d.nz & ((1u << lane) - 1u))] = lane;
  __syncwarp();
  return d;
}
// Owner lane of position k0 + lane (k0 a multiple of 32, call with the whole
// warp, for the windows k0 = 0, 32, 64, ... in order): the runs starting in
// the window mark a 32-bit mask, and the owner is the last non-empty run
// starting at or before the position. `before` counts the non-empty runs that
// start before the window (0 for the first) and is advanced past it.
__device__ __forceinline__ int deal_owner(const Deal& d, int32_t L, int32_t k0, const int32_t* comp, int lane,
                                          int& before) {
  const bool in_win = L > 0 && d.excl >= k0 && d.excl < k0 + 32;
  const unsigned M = __reduce_or_sync(0xffffffffu, in_win ? 1u << (d.excl - k0) : 0u);
  const int r = before + __popc(M & (0xffffffffu >> (31 - lane))) - 1;
  before += __popc(M);
  return comp[r < 0 ? 0 : r];
}

// The row of slot p, one of 32 consecutive slots of a warp, p0 the first (the
// whole warp calls): the warp's first and last rows by two searches of rp, the
// lane's between them.
__device__ __forceinline__ int32_t row_of_slot(int32_t n, const int32_t* __restrict__ rp, int32_t p0, int32_t p,
                                               int32_t p_last) {
  auto search = [&](int32_t lo, int32_t hi, int32_t q) {  // last row in [lo, hi] that starts at or before q
    while (lo < hi) {
      const int32_t mid = lo + ((hi - lo + 1) >> 1);
      if (rp[mid] <= q) lo = mid; else hi = mid - 1;
    }
    return lo;
  };
  const int32_t x0 = search(0, n - 1, p0);
  return search(x0, search(x0, n - 1, p_last), p);
}

}  // namespace gc
