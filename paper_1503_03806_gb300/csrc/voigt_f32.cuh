// voigt_f32.cuh -- device pieces of the FP32 form shared by its kernels: the
// method classes of a (line, point span) pair, the Gauss-Hermite terms, the
// compensated sums, and the whole-span loops.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "helk_internal.cuh"

namespace helk {

// ------------------------------------------------------------ FP32 form --
// Method classes of one (line, tile) pair.  |u| is monotone in |i - c| in
// the FP32 arithmetic used per point (u = fma(d, beta, -phi) is correctly
// rounded, so monotone in the exact integer d, and fma(u, u, a^2) is monotone
// in |u|), so the extreme r^2 over the tile's covered points decide whether
// every point of the pair uses the same method.  Pure pairs run a
// branch-free loop over all slots (independent chains the compiler can
// interleave); mixed pairs -- those containing a method boundary or the line
// core -- decide per point.
enum { CLS_GH1 = 1, CLS_GH3 = 2, CLS_MIXED = 3 };  // 0: the line misses the warp
constexpr int KAHAN_GROUP = 32;             // lines per compensated partial

// Hardware reciprocal approximation (max relative error ~1 ulp); every
// argument here is >= 100, far from the denormal range.
__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// v 2^E as a double, for a normal float v, from its bits (integer
// operations only: the conversion and scaling would otherwise be two
// operations of the FP64 unit, which runs at 1/64 of the FP32 rate here).
// Exact: the double holds v's sign and 24-bit significand at the shifted
// exponent; zero stays (signed) zero.  A subnormal v, or a result outside
// the double's normal range, takes the FP64 route.
__device__ __forceinline__ double scaled_to_double(float v, int E) {
  const unsigned b = __float_as_uint(v);
  if ((b & 0x7FFFFFFFu) == 0) return __longlong_as_double((long long)((unsigned long long)(b >> 31) << 63));
  const int ef = (int)((b >> 23) & 0xFF);
  const int e = ef - 127 + 1023 + E;
  if (ef == 0 || e <= 0 || e >= 2047) return ldexp((double)v, E);
  return __longlong_as_double((long long)(((unsigned long long)(b >> 31) << 63) |
                                          ((unsigned long long)e << 52) |
                                          ((unsigned long long)(b & 0x7FFFFF) << 29)));
}

__device__ __forceinline__ void kahan_add(float &s, float &c, float v) {
  const float y = v - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// Kahan-adds the plain partials into (sum, comp) and starts a new group.
// The loops over a group's lines run in stretches that end where the group
// is full, so the check is made once per stretch, not once per line.
template <int NSLOT>
__device__ __forceinline__ void kahan_fold(int &ngroup, float (&sum)[NSLOT], float (&comp)[NSLOT],
                                           float (&part)[NSLOT]) {
  ngroup = 0;
#pragma unroll
  for (int k = 0; k < NSLOT; ++k) {
    kahan_add(sum[k], comp[k], part[k]);
    part[k] = 0.0f;
  }
}

// 3-node Gauss-Hermite (nodes 0, +-t, t^2 = 3/2, weights 4 w1, w1):
//   (a w1/pi) [4/r2 + 2q/p],  q = r2 + t^2,  p = ((u-t)^2+a^2)((u+t)^2+a^2).
// With u^2 = r2 - a^2 both factors are polynomials in r2 alone:
//   p = r2 (r2 - 3) + C,  C = 9/4 + 6 a^2,
//   2p + q r2 = r2 (3 r2 - 9/2) + 2C,
// so the term is n / (r2 p) with n = r2 (c3 r2 + c45) + c2, the line's
// factor P3h = 2 a w1 S'/pi folded into c3 = 3 P3h, c45 = -9/2 P3h,
// c2 = 2C P3h.  No cancellation for r2 >= 100 (r2^2 >= 33 x 3 r2); FP32
// relative error < 5e-7 over 100 <= r2 < 1e6.
struct Gh3Line {
  float a2, C, c3, c45, c2;
  Gh3Line() = default;
  __device__ __forceinline__ Gh3Line(float a2_, float C_, float c3_, float c45_, float c2_)
      : a2(a2_), C(C_), c3(c3_), c45(c45_), c2(c2_) {}
  __device__ __forceinline__ Gh3Line(float a2_, float P3) {
    const float P3h = 2.0f * P3;
    a2 = a2_;
    C = fmaf(6.0f, a2_, 2.25f);
    c3 = 3.0f * P3h;
    c45 = -4.5f * P3h;
    c2 = P3h * fmaf(12.0f, a2_, 4.5f);
  }
  // numerator and denominator of the term, for the point's r2 = u^2 + a^2
  __device__ __forceinline__ void nd(float r2, float &n, float &d) const {
    const float p = fmaf(r2, r2 - 3.0f, C);
    n = fmaf(r2, fmaf(c3, r2, c45), c2);
    d = r2 * p;
  }
  // part + term
  __device__ __forceinline__ float add(float part, float r2) const {
    float n, d;
    nd(r2, n, d);
    return fmaf(n, fast_rcp(d), part);
  }
};

// The same term far from the line centre as a series in t = 1/r2:
//   n / (r2 p) = t (c3 + c45 t + c2 t^2) / (1 - 3 t + C t^2)
//              = t (g0 + g1 t + g2 t^2 + g3 t^3 + ...),
//   g0 = 3 P3h, g1 = 4.5 P3h, g2 = (11.25 - 6 a^2) P3h, g3 = (23.625 - 45 a^2) P3h
// (the product of the numerator's coefficients with those of 1/(1 - 3t +
// C t^2), e_0 = 1, e_1 = 3, e_k = 3 e_{k-1} - C e_{k-2}).  Truncated after g2,
// on r2 >= R_s with R_s >= 1000 and R_s^3 >= 1.25^3 5e7 (7.875 + 15 a^2)
// (>= 1.25^3 5e7 |g3/g0|), the relative truncation error is below 1.1e-8 for
// every a (checked in FP64 on a grid of a^2 in [0, 1e6) and r2 in [R_s, 1e6)),
// under the FP32 rounding of either form: one reciprocal and three FMAs
// instead of five FP32 operations and one reciprocal.
struct Gh3Series {
  float g0, g1, g2;
  __device__ __forceinline__ explicit Gh3Series(float a2, float P3) {
    const float P3h = 2.0f * P3;
    g0 = 3.0f * P3h;
    g1 = 4.5f * P3h;
    g2 = P3h * fmaf(-6.0f, a2, 11.25f);
  }
  // does the series hold on a span whose smallest r2 is r2near?
  static __device__ __forceinline__ bool holds(float r2near, float a2) {
    return r2near >= 1000.0f && r2near * r2near * r2near >= 9.765625e7f * fmaf(15.0f, a2, 7.875f);
  }
};

// What one warp needs of one line, prepared by one lane (lanes in parallel)
// and read by the whole warp with three broadcast loads: the kind of the
// (line, warp) pair, the covered points, the point offset, and the method's
// constants.
//   Whole-span lines (one method on every point of the warp's span: GH1, or
//   GH3 by its expansion in 1/r^2 (Gh3Series) where that holds on the whole
//   span, r^2 >= R_s; the line centre outside the span): u is stepped from the span edge
//   nearest the centre, u_k = fma(k - k_b, 32 beta, u_b), one FMA a slot (the
//   step product is exact, so each u_k is rounded once and |u_b| <= |u_k|
//   bounds its error by one ulp of u_k); d0 = (float)(base point - c) of lane
//   0, k_b = 0 (kind *_FWD, centre at or before the span) or NSLOT - 1
//   (*_BWD, centre at or after it).
//   The rest (partial cover, a method boundary, the core, the centre inside
//   the span, or GH3 nearer the centre than R_s, where the term is formed
//   exactly): d0 = (float)(wbase - c) and u = (d0 + lane + 32 k) beta
//   - phi with d0 + lane + 32 k exact, so every point's method (and whether
//   it is a core point, left to the core kernel) is decided on the same
//   correctly rounded u as in k_core_f32.
//   The series covers most of the GH3 region; the GH3 spans nearer the
//   centre run as the rest rather than in a whole-span loop of their own
//   (with one loop kind fewer the main loop's code stays within the
//   instruction caches: 0.743 against 0.763 ms a medium step).
enum { KIND_MISS = 0, KIND_GH1_FWD = 1, KIND_GH1_BWD = 2, KIND_GH3S_FWD = 3, KIND_GH3S_BWD = 4, KIND_REST = 5 };
constexpr int NKIND = 5;  // kinds after KIND_MISS

struct __align__(16) WarpLine {
  int kind;          // KIND_*
  int cls;           // CLS_* (KIND_REST)
  int lo, hi;        // covered points (grid indices; KIND_REST)
  float d0;          // point offset of lane 0 at the base slot (see above)
  float beta, nphi, a2;
  float q0, q1, q2, q3;  // GH1: P1; GH3S: g0, g1, g2 (Gh3Series); rest: P1, P3, or GH3's C, c3, c45, c2 (Gh3Line)
};

// Whole-span lines [t, t1) of one kind: GH1 or GH3 by its series, u stepped
// from the base slot.  GH1 takes one reciprocal for two slots, 1/r_a^2 =
// r_b^2 / (r_a^2 r_b^2) (5 instructions and half a reciprocal an evaluation
// instead of 4 and one: the MUFU unit, at 16 reciprocals a clock per SM, is
// the co-bound of this loop mix); the series keeps one reciprocal a slot (6
// instructions), where pairing would make the issue count the bound.
template <int NSLOT, bool FWD, bool GH3S>
__device__ __forceinline__ void span_lines(const WarpLine *wl, int t, int t1, float lanef, int &ngroup,
                                           float (&sum)[NSLOT], float (&comp)[NSLOT], float (&part)[NSLOT]) {
  while (t < t1) {
    const int te = min(t1, t + KAHAN_GROUP - ngroup);
    ngroup += te - t;
    for (; t < te; ++t) {
      const WarpLine &W = wl[t];
      const float beta = W.beta, a2 = W.a2;
      const float ub = fmaf(W.d0 + lanef, beta, W.nphi);  // u at the base slot
      const float h = 32.0f * beta;                        // u step between slots (exact)
      if (GH3S) {
        const float g0 = W.q0, g1 = W.q1, g2 = W.q2;
#pragma unroll
        for (int k = 0; k < NSLOT; ++k) {
          const float u = fmaf(FWD ? (float)k : (float)(k - (NSLOT - 1)), h, ub);
          const float rr = fast_rcp(fmaf(u, u, a2));  // t = 1/r^2 of the series
          part[k] = fmaf(rr, fmaf(fmaf(g2, rr, g1), rr, g0), part[k]);
        }
      } else {
        const float P1 = W.q0;
#pragma unroll
        for (int k = 0; k + 1 < NSLOT; k += 2) {
          const float u0 = fmaf(FWD ? (float)k : (float)(k - (NSLOT - 1)), h, ub);
          const float u1 = fmaf(FWD ? (float)(k + 1) : (float)(k + 1 - (NSLOT - 1)), h, ub);
          const float ra = fmaf(u0, u0, a2), rb = fmaf(u1, u1, a2);
          const float rr = fast_rcp(ra * rb);
          part[k] = fmaf(P1 * rb, rr, part[k]);
          part[k + 1] = fmaf(P1 * ra, rr, part[k + 1]);
        }
        if (NSLOT & 1) {
          const float u = fmaf(FWD ? (float)(NSLOT - 1) : 0.0f, h, ub);
          part[NSLOT - 1] = fmaf(P1, fast_rcp(fmaf(u, u, a2)), part[NSLOT - 1]);
        }
      }
    }
    if (ngroup == KAHAN_GROUP) kahan_fold<NSLOT>(ngroup, sum, comp, part);
  }
}

// One (line, warp) pair of a warp that owns the 32 NSLOT points from wbase,
// for one lane: the method class from the extreme r^2 over the warp's covered
// points, then the kind.  Rec: LineRec32 or a record with its wing fields.
template <int NSLOT, typename Rec>
__device__ __forceinline__ void prepare_warp_line(const Rec &L, int wbase, WarpLine &r) {
  constexpr int WSPAN = 32 * NSLOT;
  r.kind = KIND_MISS;
  const int c = L.c;
  const int lo = max(L.ilo, wbase), hi = min(L.ihi, wbase + WSPAN - 1);
  if (lo > hi) return;
  const float beta = L.beta, nphi = -L.phi_k, a2 = L.a2;
  const int dlo = lo - c, dhi = hi - c;
  const int dnear = dlo >= 1 ? dlo : (dhi <= -1 ? dhi : 0);
  const float un = fmaf((float)dnear, beta, nphi);
  const float ul = fmaf((float)dlo, beta, nphi), uh = fmaf((float)dhi, beta, nphi);
  const float r2near = fmaf(un, un, a2);
  const float r2far = fmaxf(fmaf(ul, ul, a2), fmaf(uh, uh, a2));
  const int cls = r2near >= 1.0e6f ? CLS_GH1 : ((r2near >= 100.0f && r2far < 1.0e6f) ? CLS_GH3 : CLS_MIXED);
  const bool full = (lo == wbase) && (hi == wbase + WSPAN - 1);
  r.cls = cls;
  r.lo = lo;
  r.hi = hi;
  r.beta = beta;
  r.nphi = nphi;
  r.a2 = a2;
  const bool series = cls == CLS_GH3 && Gh3Series::holds(r2near, a2);
  // (GH1 spans reach r^2 < 1e18 only: the paired reciprocals' product
  // of two r^2 stays inside the FP32 range; farther spans run as the rest)
  if (full && ((cls == CLS_GH1 && r2far < 1.0e18f) || series) && (dlo >= 0 || dhi <= 0)) {
    const bool fwd = dlo >= 0;
    r.kind = (cls == CLS_GH1 ? KIND_GH1_FWD : KIND_GH3S_FWD) + (fwd ? 0 : 1);
    r.d0 = (float)(fwd ? dlo : dhi - 31);  // lane 0 at slot 0 or NSLOT - 1
  } else {
    r.kind = KIND_REST;
    r.d0 = (float)(wbase - c);
  }
  if (series && r.kind != KIND_REST) {
    const Gh3Series gs(a2, L.P3);
    r.q0 = gs.g0;
    r.q1 = gs.g1;
    r.q2 = gs.g2;
  } else if (cls == CLS_GH3) {
    const Gh3Line g3(a2, L.P3);
    r.q0 = g3.C;
    r.q1 = g3.c3;
    r.q2 = g3.c45;
    r.q3 = g3.c2;
  } else {
    r.q0 = L.P1;
    r.q1 = L.P3;  // per-point lines form their GH3 constants when needed
  }
}

// The lanes' records (one each) ordered by kind into wl, those that miss the
// warp dropped; nk[q]: the end of kind q + 1's records (each kind then runs
// its own class-free loop).
__device__ __forceinline__ void order_warp_lines(const WarpLine &r, int lane, WarpLine *wl, int (&nk)[NKIND]) {
  unsigned b[NKIND];
#pragma unroll
  for (int q = 0; q < NKIND; ++q) b[q] = __ballot_sync(0xffffffffu, r.kind == q + 1);
  const unsigned lt = (1u << lane) - 1u;
  int pos = 0, run = 0;
#pragma unroll
  for (int q = 0; q < NKIND; ++q) {
    if (r.kind == q + 1) pos = run + __popc(b[q] & lt);
    run += __popc(b[q]);
    nk[q] = run;
  }
  if (r.kind != KIND_MISS) wl[pos] = r;
}

// Runs through a group of prepared lines (the caller has synchronised the
// warp): the whole-span kinds, then the rest -- GH1 or GH3 lines covering
// part of the span, and lines with a method boundary, their core or their
// centre in the span.
template <int NSLOT, bool COUNT>
__device__ __forceinline__ void run_warp_lines(const WarpLine *wl, const int (&nk)[NKIND], int wbase, int lane,
                                               int &ngroup, float (&sum)[NSLOT], float (&comp)[NSLOT],
                                               float (&part)[NSLOT], unsigned long long (&cnt)[4]) {
  const float lanef = (float)lane;
  span_lines<NSLOT, true, false>(wl, 0, nk[0], lanef, ngroup, sum, comp, part);
  span_lines<NSLOT, false, false>(wl, nk[0], nk[1], lanef, ngroup, sum, comp, part);
  span_lines<NSLOT, true, true>(wl, nk[1], nk[2], lanef, ngroup, sum, comp, part);
  span_lines<NSLOT, false, true>(wl, nk[2], nk[3], lanef, ngroup, sum, comp, part);
  if (COUNT) {
    cnt[2] += (unsigned long long)NSLOT * nk[1];
    cnt[1] += (unsigned long long)NSLOT * (nk[3] - nk[1]);
  }
  for (int jj = nk[3]; jj < nk[4];) {
    const int je = min(nk[4], jj + KAHAN_GROUP - ngroup);
    ngroup += je - jj;
    for (; jj < je; ++jj) {
      const WarpLine &W = wl[jj];
      const int cls = W.cls;
      const int lo = W.lo, hi = W.hi;
      const float beta = W.beta, nphi = W.nphi, a2 = W.a2;
      // (i - c) of this lane's first point, exact in FP32
      const float d0 = W.d0 + lanef;
      if (cls == CLS_GH1) {
        const float P1 = W.q0;
#pragma unroll
        for (int k = 0; k < NSLOT; ++k) {
          const int i = wbase + lane + 32 * k;
          const float u = fmaf(d0 + (float)(32 * k), beta, nphi);
          const float r2 = fmaf(u, u, a2);
          const bool in = (unsigned)(i - lo) <= (unsigned)(hi - lo);
          part[k] += in ? P1 * fast_rcp(r2) : 0.0f;
          if (COUNT) cnt[2] += in;
        }
      } else if (cls == CLS_GH3) {
        const Gh3Line g3(a2, W.q0, W.q1, W.q2, W.q3);
#pragma unroll
        for (int k = 0; k < NSLOT; ++k) {
          const int i = wbase + lane + 32 * k;
          const float u = fmaf(d0 + (float)(32 * k), beta, nphi);
          const float r2 = fmaf(u, u, a2);
          const bool in = (unsigned)(i - lo) <= (unsigned)(hi - lo);
          part[k] = in ? g3.add(part[k], r2) : part[k];
          if (COUNT) cnt[1] += in;
        }
      } else {
        // Per point: GH1 or GH3; core points (r^2 < 100) are left to the
        // core kernel (k_core_f32).  Branch-free, so the slots stay
        // independent chains: the method's numerator and denominator are
        // selected before one reciprocal (the same operations, in the same
        // order, as the whole-span loops), and the sum is kept where the
        // point is outside the window or in the core.
        const float P1 = W.q0;
        const Gh3Line g3(a2, W.q1);
#pragma unroll
        for (int k = 0; k < NSLOT; ++k) {
          const int i = wbase + lane + 32 * k;
          const float u = fmaf(d0 + (float)(32 * k), beta, nphi);
          const float r2 = fmaf(u, u, a2);
          float n, d;
          g3.nd(r2, n, d);  // not used (possibly infinite) where GH1 applies
          const bool gh1 = r2 >= 1.0e6f;
          const bool use = (unsigned)(i - lo) <= (unsigned)(hi - lo) && r2 >= 100.0f;
          const float t = fmaf(gh1 ? P1 : n, fast_rcp(gh1 ? r2 : d), part[k]);
          part[k] = use ? t : part[k];
          if (COUNT) {
            cnt[2] += use && gh1;
            cnt[1] += use && !gh1;
          }
        }
      }
    }
    if (ngroup == KAHAN_GROUP) kahan_fold<NSLOT>(ngroup, sum, comp, part);
  }
}

}  // namespace helk
