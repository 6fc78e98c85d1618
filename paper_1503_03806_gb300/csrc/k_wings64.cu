// k_wings64.cu -- the FP64 form of the interpolated-wings route (wings.cuh):
// lines taken on whole panels through 16 Chebyshev nodes, the points near the
// line centres, window edges and method boundaries one by one, and the
// Algorithm 916 cores by a polynomial in e^x.  The method of every point is
// that of the FP64 definition: the grid indices at which it changes come with
// each line (WingExt64).
//
// The FP64 unit (2 lanes a clock per SM, 1/64 of the FP32 rate) bounds all of
// it, so classes and lists are integer and FP32 work and a node or point costs
// 9 (GH1) to 15 (GH3) FP64 instructions.  1e5 lines, 3e6 points: far and cores
// 3.88 ms, near 4.09 ms, both at 86-87 % of the unit's issue rate, against 97.2 ms
// for every line at every point; 1e4 lines, 3e5 points 0.17 + 0.39 against 2.85 ms.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "helk_internal.cuh"
#include "voigt_common.cuh"
#include "wings.cuh"

namespace helk {

// 16 nodes, panels at least 5 half-widths from the poles: truncation below 6e-15
// of the profile at the closest distance, falling with its sixteenth power.
constexpr int W64_P = 16;
constexpr float W64_ETA2 = 25.0f;
constexpr int W64_CAP = 288;             // lines of a batch in shared memory
constexpr int W64_WORDS = W64_CAP / 32;
static_assert(W64_CAP >= WG_THREADS + 32, "a scan step appends up to a CTA of lines");

// tables: [side][k][16] of a child's nodes, [k][32] of a leaf's points, their
// derivatives, the nodes
constexpr int W64_TABL = 2 * W64_P * W64_P;
constexpr int W64_TABD = W64_TABL + W64_P * WG_S0;
constexpr int W64_TABT = W64_TABD + W64_P * WG_S0;
constexpr int W64_TAB = W64_TABT + W64_P;

// 1/x for x > 0: FP32 seed, then r (1 + e + e^2) with e = 1 - x r (|e| < 2^-22,
// the cube is below FP64 rounding).  Beyond the FP32 range: the division.
__device__ __forceinline__ double rcp_f64(double x) {
  float rf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"((float)x));
  if (rf == 0.0f) return 1.0 / x;
  const double r = (double)rf;
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// A line in a group's shared memory; grid indices counted from the group's
// first point, clamped to just outside the group.
struct __align__(16) WingLine64 {
  double nu0p, xh;         // shifted centre; xh + xl = nu0p - nu_min
  double ku, a2, P1;       // P1 = S' a / sqrt(pi), also the GH3 factor 6 P3
  float xl, frac, gamma, node;
  int c, ilo, ihi, g1l, g1r, g3l, g3r, pad;
};
static_assert(sizeof(WingLine64) == 96, "WingLine64 must be 96 bytes");

__device__ __forceinline__ int clamp_to(int64_t i, int gspan) { return (int)min(max(i, (int64_t)-2), (int64_t)gspan + 1); }

// Whether a line can be taken on the panel of s points from ps (positions in
// the group): in the window, one method, far enough from the poles.  From the
// integer offsets, so the same in every group; a line taken on a panel is also
// taken, by this test, on every panel inside it.
struct WingReach64 {
  float d1, d3;
  __device__ __forceinline__ WingReach64(const WingLine64 &L, float s) {
    const float hw = 0.5f * s, q = fmaf(W64_ETA2 * hw, hw, -L.gamma * L.gamma);
    d1 = q > 0.0f ? __fsqrt_rn(q) * 1.000001f : 0.0f;
    d3 = q > 0.0f ? d1 + L.node : 0.0f;
  }
  __device__ __forceinline__ bool takes(const WingLine64 &L, int ps, int pe) const {
    if (ps < L.ilo || pe > L.ihi) return false;
    const float dl = (float)(ps - L.c) - L.frac, dh = (float)(pe - L.c) - L.frac;
    const float d = 0.5f * fabsf(dl + dh);
    if (pe <= L.g1l || ps >= L.g1r) return d >= d1;
    return (pe <= L.g3l || ps >= L.g3r) && ps > L.g1l && pe < L.g1r && d >= d3;
  }
};

__device__ __forceinline__ void wing_line64(const LineRec64 &R, const WingExt64 &X, double nu_min, int64_t gbase,
                                            int gspan, WingLine64 &L) {
  L.nu0p = R.nu0p;
  L.ku = R.ku;
  L.a2 = R.a2;
  L.P1 = R.Sp * R.a * INV_SQRTPI;
  const double x = R.nu0p - nu_min, bb = x - R.nu0p;
  L.xh = x;
  L.xl = (float)((R.nu0p - (x - bb)) + (-nu_min - bb));
  L.frac = X.frac;
  L.gamma = X.gamma;
  L.node = X.node;
  L.c = X.c - (int)gbase;
  L.ilo = clamp_to((int64_t)R.ilo - gbase, gspan);
  L.ihi = clamp_to((int64_t)R.ihi - gbase, gspan);
  L.g1l = clamp_to((int64_t)X.g1l - gbase, gspan);
  L.g1r = clamp_to((int64_t)X.g1r - gbase, gspan);
  L.g3l = clamp_to((int64_t)X.g3l - gbase, gspan);
  L.g3r = clamp_to((int64_t)X.g3r - gbase, gspan);
}

// The quadrature terms (Sec. 2.4) of r2: GH1 P1 / r2; GH3 P1 n / (r2 p), with w = r2 -
// 3/2: p = r2 (r2 - 3) + 9/4 + 6 a^2 = w^2 + 6 a^2, n = r2 (r2 - 3/2) + 4 a^2 + 3/2 = p + 3/2
// w + 3/2 - 2 a^2.  a6 = 6 a^2, kn = 3/2 - 2 a^2.
__device__ __forceinline__ void gh3_nd(double r2, double a6, double kn, double &n, double &d) {
  const double w = r2 - 1.5, p = fma(w, w, a6);
  n = p + fma(1.5, w, kn);
  d = r2 * p;
}

// Adds the lines of a list to a panel's node sums: M lines at a time, one a lane
// of each of 32 / M groups of lanes, which share the 16 nodes (as list_nodes of
// the FP32 form).  cen: the panel's centre as a grid index.
template <int M>
__device__ __forceinline__ void list_nodes64(const WingLine64 *rec, const uint32_t *mask, const uint16_t *idx,
                                             int nwords, int w0, int step, uint16_t *q, int lane, const double *T,
                                             double cen, int m, double s, double dnu, double *f) {
  constexpr int NPL = W64_P * M / 32;
  const int grp = lane / M, at = lane % M;
  double acc[NPL], tn[NPL];
#pragma unroll
  for (int j = 0; j < NPL; ++j) {
    acc[j] = 0.0;
    tn[j] = T[grp * NPL + j];
  }
  const double ph = cen * dnu, pl = fma(cen, dnu, -ph), hstep = 0.5 * s * dnu;
  int n = 0;
  bool any = false;
  for (int w = w0;; w += step) {
    const bool fin = w >= nwords;  // warp-uniform
    if (!fin) {
      const uint32_t b = mask[w];
      if (b == 0) continue;
      if ((b >> lane) & 1u) {
        const int j = 32 * w + lane;
        q[n + __popc(b & ((1u << lane) - 1u))] = idx ? idx[j] : (uint16_t)j;
      }
      n += __popc(b);
      __syncwarp();
      if (n < 32) continue;
    } else if (n == 0) {
      break;
    }
    any = true;
    const int take = min(n, 32);
#pragma unroll 1
    for (int i = 0; i < take; i += M) {
      const bool have = i + at < take;
      const WingLine64 &L = rec[q[have ? i + at : 0]];
      const double ku = L.ku, a2 = L.a2, P1 = have ? L.P1 : 0.0;
      const double uc = ((ph - L.xh) + (pl - (double)L.xl)) * ku, hw = hstep * ku;
      const bool gh1 = m <= L.g1l || m >= L.g1r;  // the panel lies on one side: its middle point decides
      if (__any_sync(0xffffffffu, have && !gh1)) {
        // one reciprocal for either method: lanes of both share the pass
        const double a6 = 6.0 * a2, kn = fma(-2.0, a2, 1.5);
#pragma unroll
        for (int j = 0; j < NPL; ++j) {
          const double u = fma(tn[j], hw, uc), r2 = fma(u, u, a2);
          double nn, dd;
          gh3_nd(r2, a6, kn, nn, dd);
          acc[j] = fma(gh1 ? P1 : P1 * nn, rcp_f64(gh1 ? r2 : dd), acc[j]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < NPL; ++j) {
          const double u = fma(tn[j], hw, uc);
          acc[j] = fma(P1, rcp_f64(fma(u, u, a2)), acc[j]);
        }
      }
    }
    if (fin) break;
    n -= 32;
    const uint16_t e = q[32 + lane];
    __syncwarp();
    q[lane] = e;
    __syncwarp();
  }
  if (any) {
    double v = 0.0;
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
#pragma unroll
      for (int o = M / 2; o >= 1; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
      v = at == j ? acc[j] : v;
    }
    if (at < NPL) f[grp * NPL + at] += v;
  }
  __syncwarp();
}

enum { L64_L0 = 0, L64_L1 = 8, L64_L2 = 12, L64_U = 14, L64_N = 22 };

struct WingSmem64 {
  WingLine64 rec[W64_CAP];
  uint32_t mask[L64_N][W64_WORDS];
  uint16_t q[WG_WARPS][64];
  int wcnt[WG_WARPS];
};

// As wing_scan of the FP32 form.
template <bool UNRES, typename Work>
__device__ __forceinline__ void wing_scan64(WingSmem64 &S, const LineRec64 *__restrict__ rec,
                                            const WingExt64 *__restrict__ ext, double nu_min, int64_t first,
                                            int64_t last, int64_t stride, int64_t gbase, int64_t s, bool gok, bool ok2,
                                            bool ok1, bool ok0, int ngrid, Work work) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t gend = min(gbase + 8 * s, (int64_t)ngrid) - 1;
  const int gspan = (int)min(8 * s, (int64_t)1 << 30);
  const int nfull = (int)((gend + 1 - gbase) / s);  // panels on the grid in full
  const int is = (int)s;
  const float fs = (float)s;
  int total = 0;
  for (int64_t l0 = first; l0 < last; l0 += stride) {
    const int64_t l = l0 + tid;
    WingLine64 L;
    bool keep = false;
    if (l < last) {
      const int2 win = *reinterpret_cast<const int2 *>(&rec[l].ilo);
      if (win.x <= gend && win.y >= gbase && win.x <= win.y) {
        const WingExt64 X = ext[l];
        // lines whose whole window is core are the core kernel's
        if (!(X.g3l < win.x && X.g3r > win.y)) {
          wing_line64(rec[l], X, nu_min, gbase, gspan, L);
          keep = !(gok && WingReach64(L, 8.0f * fs).takes(L, 0, gspan - 1));
        }
      }
    }
    const unsigned b = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) S.wcnt[w] = __popc(b);
    __syncthreads();
    int at = total, n = 0;
#pragma unroll
    for (int i = 0; i < WG_WARPS; ++i) {
      const int v = S.wcnt[i];
      if (i < w) at += v;
      n += v;
    }
    if (keep) S.rec[at + __popc(b & ((1u << lane) - 1u))] = L;
    total += n;
    __syncthreads();
    if (total > W64_CAP - WG_THREADS || (total > 0 && l0 + stride >= last)) {  // CTA-uniform; total <= W64_CAP
      for (int t = 32 * w; t < total; t += WG_THREADS) {
        const bool in = t + lane < total;
        const WingLine64 &M = S.rec[min(t + lane, total - 1)];
        uint32_t mine = 0;  // lane k keeps list k's mask
        bool k2[2], k1[4];
        {
          const WingReach64 T(M, 4.0f * fs);
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            k2[p] = in && ok2 && 4 * p + 4 <= nfull && T.takes(M, 4 * p * is, 4 * (p + 1) * is - 1);
            const uint32_t m = __ballot_sync(0xffffffffu, k2[p]);
            if (lane == L64_L2 + p) mine = m;
          }
        }
        {
          const WingReach64 T(M, 2.0f * fs);
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            k1[p] = in && ok1 && 2 * p + 2 <= nfull && T.takes(M, 2 * p * is, 2 * (p + 1) * is - 1);
            const uint32_t m = __ballot_sync(0xffffffffu, k1[p] && !k2[p >> 1]);
            if (lane == L64_L1 + p) mine = m;
          }
        }
        {
          const WingReach64 T(M, fs);
#pragma unroll
          for (int p = 0; p < 8; ++p) {
            const bool up = k2[p >> 2] || k1[p >> 1];
            const bool k0 = in && !up && ok0 && p + 1 <= nfull && T.takes(M, p * is, (p + 1) * is - 1);
            uint32_t m = __ballot_sync(0xffffffffu, k0);
            if (lane == L64_L0 + p) mine = m;
            if (UNRES) {
              m = __ballot_sync(0xffffffffu,
                                in && !up && !k0 && M.ilo <= (p + 1) * is - 1 && M.ihi >= p * is);
              if (lane == L64_U + p) mine = m;
            }
          }
        }
        if (lane < (UNRES ? L64_N : L64_U)) S.mask[lane][t >> 5] = mine;
      }
      __syncthreads();
      work(total);
      total = 0;
      __syncthreads();
    }
  }
}

// ------------------------------------------------------------------ cores --
// Algorithm 916 in FP64 as a polynomial in X = e^x (the derivation stands with
// the FP32 form in voigt_core.cuh):
//   K = e^{-x^2} [ A + D sin^2(xy) + sum_n c_n (X^n + X^-n) ],  h = 1/2,
//   c_n = (h/pi) y e^{-n^2/4} / (n^2/4 + y^2).
// n up to 32 reaches A916_TAIL past x = 10; a warp sums only as far as its
// largest x needs.
constexpr int CORE64_TERMS = 32;
__device__ constexpr double CORE64_GAUSS[CORE64_TERMS] = {  // e^{-n^2/4}, n = 1 .. 32
    0x1.8ebef9eac820bp-1,   0x1.78b56362cef38p-2,   0x1.afb718e8457f7p-4,   0x1.2c155b8213cf4p-6,
    0x1.fa0e9586aebc7p-10,  0x1.02cf22526545ap-13,  0x1.411fb0da07713p-18,  0x1.e355bbaee85cbp-24,
    0x1.b93de1e27ca3bp-30,  0x1.e8a37a45fc32ep-37,  0x1.4835bd010a41bp-44,  0x1.0b6c3afdde064p-52,
    0x1.0851945bd91fcp-61,  0x1.3ce9b9de78f85p-71,  0x1.ccee1660198f4p-82,  0x1.969d47321e4ccp-93,
    0x1.b31fc898ca55ep-105, 0x1.1a6baeadb4fd1p-117, 0x1.bcb9d36e6100dp-131, 0x1.a8c1f14e2af5dp-145,
    0x1.ec1f31193575dp-160, 0x1.59d34dd8a5473p-175, 0x1.26cc2dd187404p-191, 0x1.30d759323998cp-208,
    0x1.7e63c38374debp-226, 0x1.22ee965fbfd1bp-244, 0x1.0c826832d0d94p-263, 0x1.2c9d6038f58d1p-283,
    0x1.98443e5ab2edep-304, 0x1.504d7244d31c8p-325, 0x1.500bdda2b0200p-347, 0x1.9755956ad4e9cp-370};

// e^z, |z| <= 100, as 2^m (1 + p), 1 + p rounded, what the rounding cut off in
// lo: p = expm1(r) by its Taylor polynomial to r^12 (|r| <= ln2 / 2: below 2e-16).
__device__ __forceinline__ double exp_parts(double z, int &m, double &lo) {
  const double g = fma(z, 0x1.71547652b82fep+0, 0x1.8p52), f = g - 0x1.8p52;  // nearest integer
  const double r = fma(f, -0x1.473de6af278edp-34, fma(f, -0x1.62e42fef00000p-1, z));
  double q = 1.0 / 479001600.0;
  q = fma(q, r, 1.0 / 39916800.0);
  q = fma(q, r, 1.0 / 3628800.0);
  q = fma(q, r, 1.0 / 362880.0);
  q = fma(q, r, 1.0 / 40320.0);
  q = fma(q, r, 1.0 / 5040.0);
  q = fma(q, r, 1.0 / 720.0);
  q = fma(q, r, 1.0 / 120.0);
  q = fma(q, r, 1.0 / 24.0);
  q = fma(q, r, 1.0 / 6.0);
  q = fma(q, r, 0.5);
  const double p = fma(r * r, q, r), e = 1.0 + p;
  lo = p - (e - 1.0);
  m = __double2loint(g);
  return e;
}
__device__ __forceinline__ double scale2(double v, int m) {  // v 2^m, v and the result normal
  return __hiloint2double(__double2hiint(v) + (m << 20), __double2loint(v));
}

// sin t, |t| <= pi / 2, by its Taylor polynomial to t^19 (below 3e-16)
__device__ __forceinline__ double sin_poly(double t) {
  const double z = t * t;
  double q = -1.0 / 121645100408832000.0;
  q = fma(q, z, 1.0 / 355687428096000.0);
  q = fma(q, z, -1.0 / 1307674368000.0);
  q = fma(q, z, 1.0 / 6227020800.0);
  q = fma(q, z, -1.0 / 39916800.0);
  q = fma(q, z, 1.0 / 362880.0);
  q = fma(q, z, -1.0 / 5040.0);
  q = fma(q, z, 1.0 / 120.0);
  q = fma(q, z, -1.0 / 6.0);
  return fma(q * z, t, t);
}

// K(x, y) with the line's constants; c: c_n at c[n - 1]; np, nn: terms of the
// powers of X and 1/X that the warp's points need.
__device__ __forceinline__ double k916_core64(double x, double y, double A, double D, const double *c, int np,
                                              int nn) {
  int m, mx;
  double lo, lox;
  const double x2 = x * x, ex = fma(x, x, -x2);  // x^2 = x2 + ex
  double g = exp_parts(-x2, mx, lox);
  g = scale2(g + fma(-ex, g, lox), mx);
  const double e = exp_parts(x, m, lo);
  const double r = rcp_f64(e);
  const double X = scale2(e, m), Y = scale2(r, -m);
  double p = 0.0, n = 0.0;
#pragma unroll 4
  for (int t = np - 1; t >= 0; --t) p = fma(p, X, c[t]);
#pragma unroll 2
  for (int t = nn - 1; t >= 0; --t) n = fma(n, Y, c[t]);
  p *= X;
  p = fma(p * (x + x), lo * r, p);  // X was rounded: its powers by 2x as much at the largest term
  const double xy = x * y;
  const double f = fma(xy, 0x1.45f306dc9c883p-2, 0x1.8p52) - 0x1.8p52;  // sin^2 has period pi
  const double s = sin_poly(fma(f, -0x1.0b4611a626331p-33, fma(f, -0x1.921fb54400000p+1, xy)));
  return g * (fma(s * s, D, A) + fma(n, Y, p));
}

struct __align__(16) CoreLine64 {
  double nu0p, ku, y, A, D, Sp;
  int lo, hi;
};

// The core sums of the CTA's 256 points (one a lane), as k_core_f32 does it.
__device__ __forceinline__ void core_points64(CoreLine64 (*s_line)[32], double (*s_c)[CORE64_TERMS],
                                              const LineRec64 *__restrict__ rec, const WingExt64 *__restrict__ ext,
                                              int64_t nlines, const int32_t *__restrict__ ckey, int ngrid,
                                              double nu_min, double dnu, const CondStats &cst,
                                              const int *__restrict__ cb, int64_t blk, double *__restrict__ kcore) {
  const int cw1 = cst.core_w1;
  if (cw1 == 0) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t A = blk * WG_THREADS + 32 * w;
  if (A >= ngrid) return;
  const int64_t B = min(A + 32, (int64_t)ngrid);
  int64_t W = cw1 - 1;
  if (W < CORE_BLK_PTS - 32) {  // the reach of the lines of this block and its neighbours
    const int nblk = core_blocks(ngrid), b = (int)(A / CORE_BLK_PTS);
    int r = cb[b];
    if (b > 0) r = max(r, cb[b - 1]);
    if (b + 1 < nblk) r = max(r, cb[b + 1]);
    W = r - 1;
  }
  const int64_t first = warp_search(ckey, 0, nlines, A - W, false);
  const int64_t last = warp_search(ckey, first, nlines, B - 1 + W, true);
  const int i = (int)(A + lane);
  const double nu = __dadd_rn(nu_min, __dmul_rn((double)i, dnu));
  const double gauss = CORE64_GAUSS[lane] * (0.5 * 0.31830988618379067154);  // h / pi
  const double n2 = 0.25 * (double)((lane + 1) * (lane + 1));
  double v = 0.0;
  for (int64_t l0 = first; l0 < last; l0 += 32) {
    const int64_t l = l0 + lane;
    int lo = 1, hi = 0;
    if (l < last) {
      const int2 win = *reinterpret_cast<const int2 *>(&rec[l].ilo);
      const int4 g = *reinterpret_cast<const int4 *>(&ext[l]);
      if (g.z != INT_MAX || g.w != INT_MIN) {  // a < 10
        lo = max(win.x, g.z + 1);
        hi = min(win.y, g.w - 1);
      }
    }
    uint32_t todo = __ballot_sync(0xffffffffu, lo <= hi && lo < B && hi >= A);
    if (todo == 0) continue;
    __syncwarp();
    if ((todo >> lane) & 1u) {
      const LineRec64 &R = rec[l];
      CoreLine64 q;
      q.nu0p = R.nu0p;
      q.ku = R.ku;
      q.y = R.a;
      q.A = fma(-0.31830988618379067154 * R.a, R.sig1, R.erfcx_a);
      q.D = (R.a > 1.0e-30 ? 0.31830988618379067154 / R.a : 0.0) - 2.0 * q.A;
      q.Sp = R.Sp;
      q.lo = lo;
      q.hi = hi;
      s_line[w][lane] = q;
    }
    __syncwarp();
    for (; todo; todo &= todo - 1) {
      const CoreLine64 &L = s_line[w][__ffs(todo) - 1];
      const bool in = i >= L.lo && i <= L.hi;
      const double y = L.y;
      s_c[w][lane] = gauss * y * rcp_f64(fma(y, y, n2));
      const double x = fabs(__dmul_rn(__dsub_rn(nu, L.nu0p), L.ku));
      // the terms within A916_TAIL of the warp's points: n h <= x + 6.2, and n h <=
      // 6.2 - x for the powers of 1/X
      const float xf = (float)x;
      const int tp = in ? min(CORE64_TERMS, (int)(2.0f * xf + 13.4f)) : 0, tn = in ? max(0, (int)(13.4f - 2.0f * xf)) : 0;
      const int np = __reduce_max_sync(0xffffffffu, tp), nn = __reduce_max_sync(0xffffffffu, tn);
      __syncwarp();
      if (in) v = fma(L.Sp, k916_core64(x, y, L.A, L.D, s_c[w], np, nn), v);
      __syncwarp();  // the table is rebuilt for the next line
    }
  }
  if (i < ngrid) kcore[i] = v;
}

// ---------------------------------------------------------------- kernels --
// The far kernel's CTAs (node sums of the coarser panels) first, then the core
// sums, 256 points a CTA: one launch, so that they share the GPU.  LIST: the
// conditions are those of `list` (without it the index is not kept in a register).
template <bool LIST>
__global__ void __launch_bounds__(WG_THREADS, 2)
    k_wing_far64(const LineRec64 *__restrict__ rec_all, const WingExt64 *__restrict__ ext_all, int64_t nlines,
                 const int32_t *__restrict__ ckey32, const int32_t *__restrict__ lo_all,
                 const int32_t *__restrict__ hi_all, WingGeom G, double nu_min, double dnu,
                 const int *__restrict__ list, const CondStats *__restrict__ cst, const int *__restrict__ core_blk,
                 const double *__restrict__ tab, double *__restrict__ F_all, double *__restrict__ kcore_all) {
  __shared__ WingSmem64 S;
  __shared__ double fs[WG_WARPS][3][W64_P];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cond = LIST ? list[blockIdx.y] : blockIdx.y;
  const LineRec64 *rec = rec_all + (int64_t)cond * nlines;
  const WingExt64 *ext = ext_all + (int64_t)cond * nlines;
  if ((int)blockIdx.x >= G.farblk) {
    static_assert(sizeof(S.rec) >= sizeof(CoreLine64) * WG_THREADS + sizeof(double) * WG_WARPS * CORE64_TERMS,
                  "the core CTAs use the line array");
    CoreLine64(*sl)[32] = reinterpret_cast<CoreLine64(*)[32]>(S.rec);
    double(*sc)[CORE64_TERMS] = reinterpret_cast<double(*)[CORE64_TERMS]>(sl + WG_WARPS);
    core_points64(sl, sc, rec, ext, nlines, ckey32, G.ngrid, nu_min, dnu, cst[cond],
                  core_blk + (int64_t)cond * core_blocks(G.ngrid), (int64_t)blockIdx.x - G.farblk,
                  kcore_all + (int64_t)cond * G.ngrid);
    return;
  }
  int k = G.nstage - 1, b = blockIdx.x;
  while (k > 1 && b >= G.groups[k] * G.parts[k]) b -= G.groups[k] * G.parts[k], --k;
  const int top = wing_top(G, cst[cond].wmax), l0 = wing_level(G, k);
  if (l0 > top) return;  // no window holds a panel of this stage
  const int grp = b / G.parts[k], part = b % G.parts[k];
  const int64_t s = (int64_t)WG_S0 << l0;
  const int64_t gbase = (int64_t)grp * 8 * s;
  const bool u1 = l0 + 1 <= top, u2 = l0 + 2 <= top;
  const bool gok = l0 + 3 <= top && gbase + 8 * s <= G.ngrid;
  const int64_t m = (int64_t)cond * G.nmap + G.mapoff[k] + grp;
  const int64_t first = lo_all[m] + (int64_t)part * WG_THREADS, last = hi_all[m];
  if (lane < W64_P)
    for (int v = 0; v < 3; ++v) fs[w][v][lane] = 0.0;
  __syncwarp();
  wing_scan64<false>(
      S, rec, ext, nu_min, first, last, (int64_t)G.parts[k] * WG_THREADS, gbase, s, gok, u2, u1, true, G.ngrid,
      [&](int total) {
        const int nw = (total + 31) >> 5;
#pragma unroll 1
        for (int v = 0; v < 3; ++v) {  // own panel, then a share of the coarser ones
          const int wide = 1 << v, pan = w >> v;
          const double sp = (double)(s * wide);
          list_nodes64<16>(S.rec, S.mask[(v == 0 ? L64_L0 : v == 1 ? L64_L1 : L64_L2) + pan], nullptr, nw,
                           w & (wide - 1), wide, S.q[w], lane, tab + W64_TABT,
                           (double)gbase + ((double)pan + 0.5) * sp - 0.5, (int)(((int64_t)pan * 2 + 1) * s * wide / 2),
                           sp, dnu, fs[w][v]);
        }
      });
  __syncthreads();
  double *F = F_all + (int64_t)cond * G.fslots * W64_P;
  const int np = G.parts[k];
  if (lane < W64_P) {
    const int64_t i0 = (int64_t)grp * 8 + w;
    if (i0 < G.npan[l0]) F[(G.foff[l0] + i0 * np + part) * W64_P + lane] = fs[w][0][lane];
    if (u1 && w < 4) {
      const int64_t i1 = (int64_t)grp * 4 + w;
      if (i1 < G.npan[l0 + 1])
        F[(G.foff[l0 + 1] + i1 * np + part) * W64_P + lane] = fs[2 * w][1][lane] + fs[2 * w + 1][1][lane];
    }
    if (u2 && w < 2) {
      const int64_t i2 = (int64_t)grp * 2 + w;
      if (i2 < G.npan[l0 + 2])
        F[(G.foff[l0 + 2] + i2 * np + part) * W64_P + lane] = (fs[4 * w][2][lane] + fs[4 * w + 1][2][lane]) +
                                                              (fs[4 * w + 2][2][lane] + fs[4 * w + 3][2][lane]);
    }
  }
}

// Both children of a panel at once: lanes 0 .. 15 the nodes of the lower half,
// lanes 16 .. 31 those of the upper, plus their own node sums f; the side
// `side` (or both, side < 0) is written to out.
__device__ __forceinline__ void wing_children64(const double *tab, const double *v, double f, int lane, int side,
                                                double *out) {
  const double *M = tab + (lane >> 4) * (W64_P * W64_P) + (lane & 15);
  double r = f;
#pragma unroll
  for (int k = 0; k < W64_P; ++k) r = fma(M[k * W64_P], v[k], r);
  __syncwarp();  // `out` may be v itself
  if (side < 0 || (lane >> 4) == side) out[(side < 0 ? lane >> 4 : 0) * W64_P + (lane & 15)] = r;
  __syncwarp();
}

enum { S64_H = 0, S64_L = 2, S64_G1 = 6, S64_D = 10, S64_N = 14 };
// Leaf lists up to this length are run point by point (32 points against 16 nodes
// and the list's fixed cost).
constexpr int W64_LEAF_MIN = 3;

// NL: leaves of a warp's panel, 4 or 1 (WingGeom::lvl0 2 or 0).
template <int NL, bool LIST>
__global__ void __launch_bounds__(WG_THREADS, 3)
    k_wing_near64(const LineRec64 *__restrict__ rec_all, const WingExt64 *__restrict__ ext_all, int64_t nlines,
                  const int32_t *__restrict__ lo_all, const int32_t *__restrict__ hi_all, WingGeom G, double nu_min,
                  double dnu, const int *__restrict__ list, const CondStats *__restrict__ cst,
                  const double *__restrict__ tab, const double *__restrict__ F_all,
                  const double *__restrict__ kcore_all, double weight, int accumulate,
                  double *__restrict__ kappa_all) {
  constexpr int s = NL * WG_S0, NH = NL / 2, NV = NL == 1 ? 3 : 9;
  __shared__ WingSmem64 S;
  __shared__ double fs[WG_WARPS][NV][W64_P];
  __shared__ uint16_t s_uq[WG_WARPS][W64_CAP];
  __shared__ uint32_t s_sub[WG_WARPS][S64_N][W64_WORDS];
  __shared__ double s_top[W64_P];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cond = LIST ? list[blockIdx.y] : blockIdx.y;
  const int ngrid = G.ngrid;
  const int64_t gbase = (int64_t)blockIdx.x * 8 * s;
  const int top = wing_top(G, cst[cond].wmax);
  if (lane < W64_P)
    for (int v = 0; v < NV; ++v) fs[w][v][lane] = 0.0;
  __syncwarp();
  const int64_t p0 = gbase + w * s;
  double sum[NL], nu[NL];
#pragma unroll
  for (int k = 0; k < NL; ++k) {
    sum[k] = 0.0;
    nu[k] = __dadd_rn(nu_min, __dmul_rn((double)(p0 + 32 * k + lane), dnu));
  }
  uint16_t *q = S.q[w], *uq = s_uq[w];
  uint32_t *sub = s_sub[w][0];
  const int64_t m = (int64_t)cond * G.nmap + blockIdx.x;
  const int left = (int)min((int64_t)s, (int64_t)ngrid - p0);  // points of the panel on the grid
  const int base = w * s;                                      // the panel's first point in the group
  wing_scan64<true>(
      S, rec_all + (int64_t)cond * nlines, ext_all + (int64_t)cond * nlines, nu_min, lo_all[m], hi_all[m], WG_THREADS,
      gbase, s, top >= G.lvl0 + 3 && gbase + 8 * s <= ngrid, top >= G.lvl0 + 2, top >= G.lvl0 + 1, top >= G.lvl0, ngrid,
      [&](int total) {
        const int nw = (total + 31) >> 5;
        // lines not taken on the panel: its halves, its leaves, point by point
        int n = 0;
        for (int wd = 0; wd < nw; ++wd) {
          const uint32_t b = S.mask[L64_U + w][wd];
          if ((b >> lane) & 1u) uq[n + __popc(b & ((1u << lane) - 1u))] = (uint16_t)(32 * wd + lane);
          n += __popc(b);
        }
        __syncwarp();
        const int nu32 = (n + 31) >> 5;
        int nleaf[NL];
#pragma unroll
        for (int p = 0; p < NL; ++p) nleaf[p] = 0;
#pragma unroll 1
        for (int t = 0; t < nu32; ++t) {
          const bool in = 32 * t + lane < n;
          const WingLine64 &L = S.rec[uq[in ? 32 * t + lane : 0]];
          uint32_t mine = 0;  // lane k keeps list k's mask
          const WingReach64 T1(L, 64.0f), T0(L, 32.0f);
          bool kh[2] = {false, false};
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            const int hb = base + 64 * h;
            kh[h] = in && top >= 1 && 64 * (h + 1) <= left && T1.takes(L, hb, hb + 63);
            const uint32_t mk = __ballot_sync(0xffffffffu, kh[h]);
            if (lane == S64_H + h) mine = mk;
          }
#pragma unroll
          for (int p = 0; p < NL; ++p) {
            const int pb = base + 32 * p;
            const bool rest = in && !kh[p >> 1];
            bool k0 = false;
            if (NL > 1) {
              k0 = rest && top >= 0 && 32 * (p + 1) <= left && T0.takes(L, pb, pb + 31);
              const uint32_t mk = __ballot_sync(0xffffffffu, k0);
              if (lane == S64_L + p) mine = mk;
              nleaf[p] += __popc(mk);
            }
            // point by point, unless every covered point is a core point; GH1
            // throughout where every covered point is
            const int lo = max(L.ilo, pb), hi = min(L.ihi, pb + 31);
            const bool d = rest && !k0 && lo <= hi && !(lo > L.g3l && hi < L.g3r);
            const bool g1 = d && (hi <= L.g1l || lo >= L.g1r);
            uint32_t mk = __ballot_sync(0xffffffffu, g1);
            if (lane == S64_G1 + p) mine = mk;
            mk = __ballot_sync(0xffffffffu, d && !g1);
            if (lane == S64_D + p) mine = mk;
          }
          if (lane < S64_N) sub[lane * W64_WORDS + t] = mine;
        }
        __syncwarp();
#pragma unroll 1
        for (int v = 0; v < NV; ++v) {  // own panel, pair, quarter (shared), halves, leaves
          if (v >= 5) {
            const int nl = v == 5 ? nleaf[0] : v == 6 ? nleaf[1 % NL] : v == 7 ? nleaf[2 % NL] : nleaf[3 % NL];
            if (nl <= W64_LEAF_MIN) continue;
          }
          const bool out = v < 3;
          const int wide = out ? 1 << v : 1, pan = w >> v;
          const int sp = out ? s * wide : v < 5 ? 64 : 32;
          const int ps = out ? pan * sp : base + (v < 5 ? v - 3 : v - 5) * sp;
          const uint32_t *mk = out ? S.mask[(v == 0 ? L64_L0 : v == 1 ? L64_L1 : L64_L2) + pan]
                                   : sub + (v < 5 ? S64_H + v - 3 : S64_L + v - 5) * W64_WORDS;
          list_nodes64<8>(S.rec, mk, out ? nullptr : uq, out ? nw : nu32, out ? w & (wide - 1) : 0, wide, q, lane,
                          tab + W64_TABT, (double)gbase + (double)ps + 0.5 * (double)sp - 0.5, ps + sp / 2, (double)sp,
                          dnu, fs[w][v]);
        }
#pragma unroll 1
        for (int p = 0; p < NL; ++p) {
          const int ip = base + 32 * p + lane;
          const double nui = p == 0 ? nu[0] : p == 1 ? nu[1 % NL] : p == 2 ? nu[2 % NL] : nu[3 % NL];
          const bool few =
              NL > 1 && (p == 0 ? nleaf[0] : p == 1 ? nleaf[1 % NL] : p == 2 ? nleaf[2 % NL] : nleaf[3 % NL]) <= W64_LEAF_MIN;
          double part = 0.0;
#pragma unroll 1
          for (int t = 0; t < nu32; ++t) {
            const uint32_t m1 = sub[(S64_G1 + p) * W64_WORDS + t];
            const uint32_t md = sub[(S64_D + p) * W64_WORDS + t] | (few ? sub[(S64_L + p) * W64_WORDS + t] : 0u);
            if ((m1 | md) == 0) continue;
            const int n1 = __popc(m1), nd = __popc(md);
            const uint32_t lt = (1u << lane) - 1u;
            if ((m1 >> lane) & 1u) q[__popc(m1 & lt)] = uq[32 * t + lane];
            if ((md >> lane) & 1u) q[n1 + __popc(md & lt)] = uq[32 * t + lane];
            __syncwarp();
#pragma unroll 2
            for (int i = 0; i < n1; ++i) {
              const WingLine64 &D = S.rec[q[i]];
              const double u = (nui - D.nu0p) * D.ku;
              const double v = fma(D.P1, rcp_f64(fma(u, u, D.a2)), part);
              part = ip >= D.ilo && ip <= D.ihi ? v : part;
            }
#pragma unroll 1
            for (int i = n1; i < n1 + nd; ++i) {
              const WingLine64 &D = S.rec[q[i]];
              const double a2 = D.a2, P1 = D.P1;
              const double u = (nui - D.nu0p) * D.ku, r2 = fma(u, u, a2);
              const bool in = ip >= D.ilo && ip <= D.ihi, gh1 = ip <= D.g1l || ip >= D.g1r;
              const bool core = ip > D.g3l && ip < D.g3r;  // left to the core sums
              double nn = 1.0, dd = r2;
              if (__any_sync(0xffffffffu, in && !gh1 && !core)) {
                gh3_nd(r2, 6.0 * a2, fma(-2.0, a2, 1.5), nn, dd);
                nn = gh1 ? 1.0 : nn;
                dd = gh1 ? r2 : dd;
              }
              const double v = fma(P1 * nn, rcp_f64(dd), part);
              part = in && !core ? v : part;
            }
            __syncwarp();
          }
          if (p == 0) sum[0] += part;
          else if (p == 1) sum[1 % NL] += part;
          else if (p == 2) sum[2 % NL] += part;
          else sum[3 % NL] += part;
        }
      });
  __syncthreads();  // the batch's shared memory is free
  double *tv = reinterpret_cast<double *>(S.rec) + w * (9 * W64_P);
  if (top >= 0 && w == 0) {
    // the values at the nodes of the group's own panel from the
    // coarser levels, coarsest first
    const double *F = F_all + (int64_t)cond * G.fslots * W64_P;
    if (lane < W64_P) s_top[lane] = 0.0;
    __syncwarp();
    for (int l = top; l >= wing_level(G, 1); --l) {
      const int64_t p = gbase >> (5 + l);  // WG_S0 2^l points a panel
      if (p >= G.npan[l]) continue;        // not on the grid in full: nor is any coarser one
      const int np = G.parts[(l - G.lvl0) / 3];
      const double *Fp = F + (G.foff[l] + p * np) * W64_P + (lane & 15);
      double f = 0.0;
      for (int i = 0; i < np; ++i) f += Fp[i * W64_P];
      wing_children64(tab, s_top, f, lane, (int)(p & 1), s_top);
    }
  }
  __syncthreads();
  if (p0 >= ngrid) return;
  if (top >= 0) {
    // down the tree: the quarter, the pair, the warp's panel, its halves, its leaves
    const int j = lane & 15, h4 = w & 4, h2 = w & 6, side = lane >> 4;
#pragma unroll 1
    for (int t = 0; t < (NL == 1 ? 3 : 6); ++t) {
      const double f = t == 0 ? (fs[h4][2][j] + fs[h4 + 1][2][j]) + (fs[h4 + 2][2][j] + fs[h4 + 3][2][j])
                       : t == 1 ? fs[h2][1][j] + fs[h2 + 1][1][j]
                                : fs[w][(t == 2 ? 0 : t == 3 ? 3 + side : t == 4 ? 5 + side : 7 + side) % NV][j];
      // tv: quarter, pair, own; 3, 4: halves; 5 .. 8: leaves
      wing_children64(tab, t == 0 ? s_top : tv + (t - 1) * W64_P, f, lane,
                      t == 0 ? (w >> 2) & 1 : t == 1 ? (w >> 1) & 1 : t == 2 ? w & 1 : -1,
                      tv + (t < 3 ? t : t == 3 ? 3 : t == 4 ? 5 : 7) * W64_P);
    }
  }
  const bool core = cst[cond].core_w1 != 0;
  const double *kcore = kcore_all + (int64_t)cond * ngrid;
  double *kappa = kappa_all + (int64_t)cond * ngrid;
  const double rstep = 1.0 / (16.0 * dnu);
#pragma unroll 1
  for (int p = 0; p < NL; ++p) {
    const int64_t i = p0 + 32 * p + lane;
    double v = p == 0 ? sum[0] : p == 1 ? sum[1 % NL] : p == 2 ? sum[2 % NL] : sum[3 % NL];
    if (top >= 0) {
      const double *tl = tv + (NL == 1 ? 2 : 5 + p) * W64_P, *Lm = tab + W64_TABL + lane, *Ld = tab + W64_TABD + lane;
      double far = 0.0, der = 0.0;
#pragma unroll
      for (int k = 0; k < W64_P; ++k) {
        far = fma(Lm[k * WG_S0], tl[k], far);
        der = fma(Ld[k * WG_S0], tl[k], der);
      }
      // the point's wavenumber is a rounded number: its distance from the ideal
      // grid, times the derivative
      const double x = (double)i, pr = x * dnu, e1 = fma(x, dnu, -pr);
      const double nui = p == 0 ? nu[0] : p == 1 ? nu[1 % NL] : p == 2 ? nu[2 % NL] : nu[3 % NL];
      const double bb = nui - nu_min, e2 = (nu_min - (nui - bb)) + (pr - bb);
      v += fma(der, -(e1 + e2) * rstep, far);
    }
    if (i < ngrid) {
      if (core) v += kcore[i];
      v *= weight;
      kappa[i] = accumulate ? kappa[i] + v : v;
    }
  }
}

// ----------------------------------------------------------------- launch --
helk_status ensure_wing64(helk_ctx *c, int n_cond, const WingGeom &g) {
  const int64_t nl = std::max<int64_t>(c->nlines, 1);
  helk_status st = ensure_buf(c, (void **)&c->wingF, &c->wingF_cap,
                              std::max<int64_t>(1, g.fslots) * n_cond * W64_P * 8, "wing sums");
  if (st == HELK_OK)
    st = ensure_buf(c, (void **)&c->ext64, &c->ext64_cap, nl * n_cond * (int64_t)sizeof(WingExt64), "line records");
  if (st == HELK_OK) st = ensure_buf(c, (void **)&c->ckey32, &c->ckey32_cap, nl * 4, "line keys");
  if (st == HELK_OK)
    st = ensure_buf(c, (void **)&c->core_blk, &c->core_blk_cap, (int64_t)core_blocks(g.ngrid) * n_cond * 4,
                    "core reach");
  if (st == HELK_OK)
    st = ensure_buf(c, (void **)&c->kcore64, &c->kcore64_cap, (int64_t)g.ngrid * n_cond * 8, "core sums");
  if (st != HELK_OK || c->wing_tab64) return st;
  std::vector<double> t;
  wing_tables(W64_P, W64_P, t);  // children, leaf points, nodes
  std::vector<double> tab(W64_TAB);
  std::copy(t.begin(), t.begin() + W64_TABD, tab.begin());
  std::copy(t.begin() + W64_TABD, t.end(), tab.begin() + W64_TABT);
  // derivatives of the nodes' basis at the leaf's points
  const double *tn = tab.data() + W64_TABT;
  for (int i = 0; i < WG_S0; ++i) {
    const double x = (2.0 * i + 1.0 - WG_S0) / WG_S0;
    for (int k = 0; k < W64_P; ++k) {
      double d = 0.0;  // sum over j != k of prod_{l != k, j} (x - t_l) / prod_{l != k} (t_k - t_l)
      for (int j = 0; j < W64_P; ++j) {
        if (j == k) continue;
        double p = 1.0 / (tn[k] - tn[j]);
        for (int l = 0; l < W64_P; ++l)
          if (l != k && l != j) p *= (x - tn[l]) / (tn[k] - tn[l]);
        d += p;
      }
      tab[W64_TABD + (size_t)k * WG_S0 + i] = d;
    }
  }
  double *p = nullptr;
  st = cuda_check(c, cudaMalloc((void **)&p, tab.size() * 8), "wing tables");
  if (st != HELK_OK) return st;
  // on the context's stream and waited for, so that every stream finds it complete
  st = cuda_check(c, cudaMemcpyAsync(p, tab.data(), tab.size() * 8, cudaMemcpyHostToDevice, c->stream), "wing tables");
  if (st == HELK_OK) st = cuda_check(c, cudaStreamSynchronize(c->stream), "wing tables");
  if (st == HELK_OK)
    c->wing_tab64 = p;
  else
    cudaFree(p);
  return st;
}

cudaError_t launch_wing_far64(helk_ctx *c, int n_cond, const int *list, const WingGeom &g, const helk_grid &grid) {
  ++c->launches;
  const int64_t blocks = g.farblk + (grid.n + WG_THREADS - 1) / WG_THREADS;
  auto far = list ? k_wing_far64<true> : k_wing_far64<false>;
  far<<<dim3((unsigned)blocks, n_cond), WG_THREADS, 0, c->stream>>>(
      c->rec64, c->ext64, c->nlines, c->ckey32, c->tile_lo, c->tile_hi, g, grid.nu_min, grid.dnu, list,
      c->cstats, c->core_blk, c->wing_tab64, (double *)c->wingF, c->kcore64);
  return cudaGetLastError();
}

cudaError_t launch_wing_near64(helk_ctx *c, int n_cond, const int *list, const WingGeom &g, const helk_grid &grid,
                               const helk_opts &o, double *kappa) {
  ++c->launches;
  auto near = g.lvl0 == 2 ? (list ? k_wing_near64<4, true> : k_wing_near64<4, false>)
                          : (list ? k_wing_near64<1, true> : k_wing_near64<1, false>);
  near<<<dim3((unsigned)g.groups[0], n_cond), WG_THREADS, 0, c->stream>>>(
      c->rec64, c->ext64, c->nlines, c->tile_lo, c->tile_hi, g, grid.nu_min, grid.dnu, list, c->cstats,
      c->wing_tab64, (const double *)c->wingF, c->kcore64, o.weight, o.accumulate, kappa);
  return cudaGetLastError();
}

}  // namespace helk
