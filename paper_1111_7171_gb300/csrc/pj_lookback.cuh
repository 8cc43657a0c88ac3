// Decoupled look-back (D. Merrill and M. Garland, 2016): the running sum over
// the tiles before a tile, found while those tiles are still at work.  A tile's status word holds its own
// sum as soon as it is known, and later the sum over all tiles up to it.
// Word: 2 flag bits on top, the value below; written and read as one 64-bit
// access, so flag and value always belong together.  The words are zero
// before the launch.
//
// No wait is open-ended: a tile that has not published after LB_POLLS polls
// is summed again from its input, which the kernel only reads, by whoever
// waits for it.  So every launch ends, with the same result, in whatever
// order its blocks run.
#pragma once

#include "pj_common.cuh"

namespace pj {

constexpr unsigned long long LB_SUM = 1ull << 62;     // the tile's own sum
constexpr unsigned long long LB_PREFIX = 2ull << 62;  // the sum of all tiles up to it
constexpr unsigned long long LB_VALUE = (1ull << 62) - 1;
#ifndef PJ_LB_POLLS  // a test compiles with 0: every tile that is not done yet is summed again
#define PJ_LB_POLLS (1 << 12)
#endif
constexpr int LB_POLLS = PJ_LB_POLLS;

__device__ __forceinline__ unsigned long long lb_load(const unsigned long long* p) {
  return *reinterpret_cast<const volatile unsigned long long*>(p);
}
__device__ __forceinline__ void lb_store(unsigned long long* p, unsigned long long v) {
  *reinterpret_cast<volatile unsigned long long*>(p) = v;
}

// The sum over the tiles before `tile`, by one whole warp, 32 tiles a step.
// tile_sum(p): tile p's sum from its input, called by the whole warp with
// the same p; every lane returns the sum.
template <class TileSum>
__device__ __forceinline__ unsigned long long lookback_warp(const unsigned long long* status, unsigned tile,
                                                            TileSum tile_sum) {
  const int lane = threadIdx.x & 31;
  unsigned long long before = 0;
  for (long long hi = (long long)tile - 1; hi >= 0; hi -= 32) {
    const long long p = hi - lane;
    unsigned long long s = p >= 0 ? lb_load(status + p) : LB_PREFIX;
    for (int poll = 0; poll < LB_POLLS && __any_sync(FULL, (s >> 62) == 0); ++poll)
      if ((s >> 62) == 0) s = lb_load(status + p);
    unsigned missing = __ballot_sync(FULL, (s >> 62) == 0);
    while (missing) {
      const int b = __ffs((int)missing) - 1;
      missing &= missing - 1;
      const unsigned long long v = tile_sum((unsigned)(hi - b));
      if (lane == b) s = LB_SUM | v;
    }
    const unsigned done = __ballot_sync(FULL, (s >> 62) == 2);
    const int last = done ? __ffs((int)done) - 1 : 31;
    before += warp_sum(lane <= last ? s & LB_VALUE : 0ull);
    if (done) break;
  }
  return before;
}

}  // namespace pj
