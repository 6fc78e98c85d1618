// route.cuh -- the rules by which an opacity call takes interpolated wings or the
// point-by-point kernels, and one core kernel or the other (host side; needs no other
// header, so that a test can compile it alone).
#pragma once

#include <stdint.h>

#include <algorithm>
#include <cmath>

namespace helk {

// Centres of the ordered list at LIST_CUTS + 1 evenly spaced places ((n - 1) i /
// LIST_CUTS), the first and the last line among them: how many lines lie where.
constexpr int LIST_CUTS = 64;
struct ListShape {
  int64_t n;
  double at[LIST_CUTS + 1];
};

// Lines below wavenumber x, between two cuts by interpolation.
inline double lines_below(const ListShape &L, double x) {
  if (L.n <= 0 || x <= L.at[0]) return 0.0;
  if (x > L.at[LIST_CUTS]) return (double)L.n;
  const int i = (int)(std::lower_bound(L.at, L.at + LIST_CUTS + 1, x) - L.at);  // at[i - 1] < x <= at[i]
  const double f = (x - L.at[i - 1]) / (L.at[i] - L.at[i - 1]);
  return ((double)(i - 1) + f) / LIST_CUTS * (double)L.n;
}

// Lines within `reach` points of a stretch of `points` grid points, the mean over
// stretches at eight places of the grid.
inline double lines_near(const ListShape &L, double nu_min, double dnu, int64_t n, double points, double reach) {
  double sum = 0.0;
  const double w = 0.5 * std::min(points, (double)n);
  for (int k = 0; k < 8; ++k) {
    const double mid = w + ((double)n - 2.0 * w) * (k + 0.5) / 8.0;
    sum += lines_below(L, nu_min + (mid + w + reach) * dnu) - lines_below(L, nu_min + (mid - w - reach) * dnu);
  }
  return sum / 8.0;
}

// FP64 form.  Windows of at most `most` points to a side, by the cutoff alone; `half`:
// of a condition (under a Lorentz cutoff its windows may be much narrower).  The
// wings' map, tree and core pass cost the same for few lines (0.14 ns a point and ~20
// us), the direct kernel a tile of 2048 points some us a line that has a point of it:
// the wings pay from about six lines a tile on, on short grids, where the launches
// count, from about thirty.  us, wings / direct:
//   half a window of h points, 1e5 lines on 3e6 points   h = 24 2370 / 9110   64 3660 / 16000
//   3e3 lines on 2e4 points                              h = 24   77 / 154
//   3e6 points, lines a tile   2.3 (1e3 lines, h = 2500) 774 / 578    7 (1e4, h = 30) 749 / 1126
//                              17 (1e3, h = 25000) 866 / 2084
//   3e5 points                 2.3 (100, h = 2500) 175 / 121     7 (1e3, h = 30) 165 / 201
//   3e4 points                 8.5 (100, h = 250) 62 / 42       21 (300, h = 30) 68 / 61
//                              23 (100, h = 2500) 84 / 85       85 (1e3, h = 250) 95 / 117
//   3e3 points                 25 (30, h = 250) 61 / 51         85 (100, h = 250) 68 / 92
//   300 points, 10 lines 55 / 48, 100 lines 100 / 247
// Lorentz cutoff, 3e6 points, 1e5 lines (2 h of them have a point, 68 a tile)
//   h = 0.0002 (1e-7 atm) 288 / 133    0.02 318 / 251    0.2 484 / 1031    22 1930 / 6570
constexpr double WING64_MIN_HALF = 24.0;
inline bool wings_pay64(const ListShape &L, double nu_min, double dnu, int64_t n, double most, double half) {
  const double s = 1.4e5 / (double)n;
  return most >= WING64_MIN_HALF && lines_near(L, nu_min, dnu, n, 2048.0, half) * std::min(1.0, 2.0 * half) >=
                                        6.5 + std::min(25.0, s * s);
}

// FP32 form.  `most` as above; num_sms SMs.  By the lines that reach a tile of 2048
// points, too: the direct kernel's time follows them, while the wings cost some 30 us
// on short grids, 60 to 130 us on 3e6 points whatever the lines; between, grids whose
// panels are the short ones (WingGeom::lvl0 0) take the longest to pay.  us, wings /
// direct, at lines a tile (lines, half a window in points):
//   3e3 points  30 (30, 2500) 47 / 39     85 (100, 250) 42 / 43    100 (100, 2500) 46 / 50
//   3e4 points  23 (100, 2500) 46 / 39    85 (1e3, 250) 48 / 46    230 (1e3, 2500) 54 / 62
//   3e5 points  70 (3e3, 2500) 73 / 55   170 (1e3, 25000) 72 / 61  235 (1e4, 2500) 82 / 80
//              520 (3e3, 25000) 83 / 92  850 (1e5, 250) 133 / 200
//   3e6 points  52 (3e3, 25000) 197 / 136 85 (1e5, 250) 278 / 252  119 (1e5, 768) 301 / 306
//              173 (1e4, 25000) 218 / 265 235 (1e5, 2500) 325 / 406  725 (1e6, 64) 980 / 1200
constexpr double WING32_MIN_HALF = 64.0;
inline bool wings_pay32(const ListShape &L, double nu_min, double dnu, int64_t n, double most, int num_sms) {
  const double lines = n <= (int64_t)512 * num_sms ? 100.0 : n < (int64_t)2048 * num_sms ? 200.0 : 120.0;
  return most >= WING32_MIN_HALF && lines_near(L, nu_min, dnu, n, 2048.0, most) >= lines;
}

// FP32 form.  Largest beta (grid steps in Doppler units) of a line whose cores are
// taken through nodes, and whether a line of a condition can have one as small: kc is
// sqrt(ln2) nu / Gamma_D for the call's mass, or for 1 amu where the lines have masses,
// of which mass_min is the smallest (beta grows with its root; pass 1 otherwise); a
// factor of 2 for centres beyond the grid's end and for shifts.  If none can, the kernel
// without nodes gives the same sums in less time (1e5 lines with masses, 3e6 points at
// 0.01, 0.1 atm: 276 us a call, 289 with the other).
constexpr double CORE_NODE_BETA = 0.3 / 16.0;
inline bool core_nodes_possible(double nu_min, double dnu, int64_t n, double kc, double mass_min) {
  const double top = std::max(std::fabs(nu_min), std::fabs(nu_min + dnu * (double)n));
  return dnu * kc * std::sqrt(mass_min) <= 2.0 * CORE_NODE_BETA * top;
}

}  // namespace helk
