// sort_runs.cuh -- the order of a line list that is a few ordered runs one after
// the other (one species or file each).
#pragma once

#include <stdint.h>

namespace helk {

constexpr int SORT_RUNS = 16;  // runs that are told apart

// Upload: a list of ordered runs is merged or sorted.  A merge's time grows with the runs
// (each line looks for its place in every other), the radix passes' does not, and the
// latter gain on the former with the length.  In us, merged / sorted:
//   lines     8 runs       9           10          12          16
//   2.6e5    216 / 431   234 / 434   249 / 435   282 / 430   325 / 435
//   4e5      315 / 478   340 / 476   371 / 479   417 / 479   508 / 475
//   8e5      549 / 741   601 / 741   658 / 741   745 / 737   929 / 740
//   1.5e6    988 / 1206  1095 / 1206 1202 / 1208 1352 / 1205 1759 / 1208
//   5e6     3233 / 3649  3601 / 3647 3836 / 3645 4566 / 3651 6022 / 3647
//   1e7     6543 / 7020  7365 / 7020             16 runs: 12400 / 7020
// so up to 8 runs are merged at every length, and above that as many more as the length
// leaves room for.
constexpr int MERGE_RUNS = 8;
constexpr int64_t MERGE_MORE = 3000000;
inline bool merge_pays(int64_t n, int runs) {
  return runs <= MERGE_RUNS || (runs <= SORT_RUNS && (runs - MERGE_RUNS) * n <= MERGE_MORE);
}

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
