// split_ranges.h -- the rule by which the planner cuts a class into warp ranges,
// in its plain form over a prefix sum of every segment's cost.  The library
// finds the same cuts a chunk at a time (csrc/seg_walk.h); the tests compare
// the two.
#pragma once

#include <cstdint>

// bnd[w], w = 0..Wq: the segment where warp w's range starts, given the cost
// prefix cost(s) of segments [0, s) for s = 0..n (nondecreasing): the last
// boundary whose prefix is at most w / Wq of the total (bnd[0] = 0 even if
// the first segments cost nothing, bnd[Wq] = n).  With unit costs this is
// floor(n * w / Wq).
template <class Prefix>
inline void split_ranges(const Prefix& cost, uint64_t n, uint64_t Wq, uint64_t* bnd) {
  const unsigned __int128 total = cost(n);
  uint64_t s = 0;
  bnd[0] = 0;
  for (uint64_t w = 1; w <= Wq; ++w) {
    const unsigned __int128 target = total * w;
    while (s < n && static_cast<unsigned __int128>(cost(s + 1)) * Wq <= target) ++s;
    bnd[w] = s;
  }
}
