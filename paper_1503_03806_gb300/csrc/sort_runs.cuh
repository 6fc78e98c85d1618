// sort_runs.cuh -- the order of a line list that is a few ordered runs one after
// the other (one species or file each).
#pragma once

#include <stdint.h>

namespace helk {

// Upload: lists of at most SORT_RUNS ordered runs are merged, others sorted; lists of
// more than MERGE_SHORT lines if they have at most MERGE_RUNS_LONG runs.
constexpr int SORT_RUNS = 16, MERGE_RUNS_LONG = 8;
constexpr int64_t MERGE_SHORT = (int64_t)1 << 18;

struct SortRuns {
  int n, end[SORT_RUNS + 1];
};

// The place of element l in the order: its place in its run plus, in every other
// run, the number of elements before it (equal centres: earlier runs first, so the
// order is stable), by bisection, a chain of dependent loads.  nu0(i): the centre
// of element i.  Indices are 64-bit: the sum of two reaches 2^32.
template <typename Nu0>
__host__ __device__ __forceinline__ int64_t merged_place(const SortRuns &R, int64_t l, Nu0 nu0) {
  const double v = nu0(l);
  int64_t at = 0, b = 0;
  for (int r = 0; r < R.n; ++r) {
    const int64_t e = R.end[r];
    if (l >= b && l < e) {
      at += l - b;
    } else {
      int64_t lo = b, hi = e;
      const bool before = e <= l;
      while (lo < hi) {
        const int64_t m = lo + ((hi - lo) >> 1);
        const double w = nu0(m);
        if (before ? w <= v : w < v) lo = m + 1;
        else hi = m;
      }
      at += lo - b;
    }
    b = e;
  }
  return at;
}

}  // namespace helk
