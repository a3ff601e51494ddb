// Searches in ascending arrays of up to 2^31 entries (row starts), written so
// that a host program can follow every index they probe.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GM_HD __host__ __device__ __forceinline__
#else
#define GM_HD inline
#endif

namespace gm {

// Largest i in [0, n) whose entry is at or below the value sought, given that
// entry 0 is, by `threads` probes a step: count(lo, len, step) is the number
// of probes lo + t * step, t < threads with t * step < len, whose entry is (a
// prefix of them).  64 bits throughout: len + threads - 1 and t * step pass
// 2^31 for n close to it.
template <class Count>
GM_HD int64_t last_by_probes(int64_t n, int threads, Count count) {
  int64_t lo = 0, len = n;
  while (len > 1) {
    const int64_t step = (len + threads - 1) / threads;
    const int cnt = count(lo, len, step);
    const int64_t skip = cnt > 0 ? (cnt - 1) * step : 0;
    lo += skip;
    len = step < len - skip ? step : len - skip;
  }
  return lo;
}

// The same by bisection over [lo, hi), given that `at_or_below(lo)`.
template <class Index, class Pred>
GM_HD Index last_by_bisection(Index lo, Index hi, Pred at_or_below) {
  while (hi - lo > 1) {
    const Index mid = lo + (hi - lo) / 2;
    if (at_or_below(mid)) lo = mid;
    else hi = mid;
  }
  return lo;
}

}  // namespace gm
