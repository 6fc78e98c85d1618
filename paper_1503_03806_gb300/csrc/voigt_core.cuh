// voigt_core.cuh -- device functions of Algorithm 916 shared by the Voigt
// kernels and the surrogate's training-target kernel.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "helk_internal.cuh"

namespace helk {

// ------------------------------------------------------------------------
// Algorithm 916 (Sec. 2.4), FP64.  K(x, y) for 0 <= x, x^2 + y^2 < 100:
//   K = e^{-x^2} erfcx(y) cos(2xy) + (2hx/pi) e^{-x^2} sin(xy) sinc(xy)
//     + (2h/pi) [ -y cos(2xy) e^{-x^2} S1 + (y/2)(S2 + S3) ],
//   S1 = sum e^{-(nh)^2}/((nh)^2+y^2)  (per line: sig1),
//   S2 + S3 = sum (e^{-(nh+x)^2} + e^{-(nh-x)^2}) / ((nh)^2 + y^2),
// the exponentials of S2/S3 advanced by the exact ratio recurrences
//   e^{-((n+1)h -+ x)^2} = e^{-(nh -+ x)^2} * R,  R <- R e^{-2h^2}.
// Only the terms within A916_TAIL of the Gaussian peaks are summed.
static __device__ __forceinline__ void a916_range(double x, int &n0, int &n1) {
  n0 = (int)floor((x - A916_TAIL) / A916_H);
  if (n0 < 1) n0 = 1;
  n1 = (int)ceil((x + A916_TAIL) / A916_H);
}

static __device__ __noinline__ double k916_f64(double x, double y, double erfcx_y, double sig1) {
  const double h = A916_H;
  const double ex2 = exp(-(x * x));
  const double xy = x * y;
  double s, c;
  sincos(xy, &s, &c);
  const double sinc = (xy == 0.0) ? 1.0 : s / xy;
  const double c2xy = c * c - s * s;
  int n0, n1;
  a916_range(x, n0, n1);
  const double q = 0.60653065971263342360;  // e^{-2h^2}
  const double nh = n0 * h;
  const double dm = nh - x, dp = nh + x;
  double E3 = exp(-(dm * dm));
  double R3 = exp(-(2.0 * h * dm + h * h));
  double E2 = exp(-(dp * dp));
  double R2 = exp(-(2.0 * h * dp + h * h));
  double s23 = 0.0;
  const double y2 = y * y;
  for (int n = n0; n <= n1; ++n) {
    const double nhn = n * h;
    s23 += (E2 + E3) / (nhn * nhn + y2);
    E3 *= R3;
    R3 *= q;
    E2 *= R2;
    R2 *= q;
  }
  double K = ex2 * erfcx_y * c2xy;
  K += (2.0 * h / PI) * x * ex2 * s * sinc;
  K += (2.0 * h / PI) * (0.5 * y * s23 - y * c2xy * ex2 * sig1);
  return K;
}

// Algorithm 916 in FP32 for one line (y fixed), 0 <= x, x^2 + y^2 < 100.
//
// The counting variant counts the terms of the series within A916_TAIL_F32 of
// the Gaussian peaks (each dropped term is below e^{-18.49} = 9.3e-9 of its
// weight).
constexpr float A916_TAIL_F32 = 4.3f;
// n in [2(x - 4.3), 2(x + 4.3)], an interval of length 17.2: at most 18 terms
constexpr int A916_TERMS_F32 = 18;

static __device__ __forceinline__ void a916_range_f32(float x, int &n0, int &n1) {
  n0 = (int)ceilf((x - A916_TAIL_F32) * 2.0f);
  if (n0 < 1) n0 = 1;
  n1 = (int)floorf((x + A916_TAIL_F32) * 2.0f);
}

// e^{-t^2/4}, t = 0 .. A916_TERMS_F32 - 1, rounded to FP32.
__device__ constexpr float A916_GAUSS_F32[A916_TERMS_F32] = {
    0x1.0p+0f,        0x1.8ebefap-1f,   0x1.78b564p-2f,   0x1.afb718p-4f,   0x1.2c155cp-6f,
    0x1.fa0e96p-10f,  0x1.02cf22p-13f,  0x1.411fb0p-18f,  0x1.e355bcp-24f,  0x1.b93de2p-30f,
    0x1.e8a37ap-37f,  0x1.4835bep-44f,  0x1.0b6c3ap-52f,  0x1.085194p-61f,  0x1.3ce9bap-71f,
    0x1.ccee16p-82f,  0x1.969d48p-93f,  0x1.b31fc8p-105f};
// 2^{4 t} e^{-t^2/4}, t = 18 .. 22
__device__ constexpr float A916_GAUSS_HIGH[5] = {0x1.1a6baep-45f, 0x1.bcb9d4p-55f, 0x1.a8c1f2p-65f,
                                                 0x1.ec1f32p-76f, 0x1.59d34ep-87f};

// With h = 1/2 the factors of the series' terms are powers of X = e^x,
//   e^{-(nh -+ x)^2} = e^{-x^2} e^{-n^2/4} X^{+-n},
// and the closing terms need s = sin(xy) alone (cos 2xy = 1 - 2 s^2,
// x sin(xy) sinc(xy) = s^2 / y), so
//   K = e^{-x^2} [ A + D s^2 + sum_{n=1}^{22} c_n (X^n + X^-n) ],
//   A = erfcx(y) - (2h/pi) y S1(y),  D = (2h/pi)/y - 2 A,
//   c_n = (h/pi) y e^{-n^2/4} / (n^2/4 + y^2),
// one FMA a term (the X^-n are below FP32 past n = 8).  Taken for x^2 <
// core_inner(y) <= 41: 22 terms reach 4.3 past x.  The powers of X double its
// relative error by 2x at the largest term, so the part that its rounding
// cut off is carried along (eps).  The c_n are kept as 2^{4n} c_n, used with
// 2^{-4} X^{+-1}, all within the FP32 range.
constexpr int CORE_TERMS = 22;
constexpr int CORE_TERMS_NEG = 8;

// The bound on x^2 between the two forms.  Outside, the 8-node Gauss-Hermite
// rule is within 3e-8 of K, up to the e^{-x^2} that it lacks (< 2e-8 of K at
// the bound for y >= 1e-8; added below that).  Checked against the exact w(z).
static __device__ __forceinline__ float core_inner(float y) {
  if (y >= 4.5f) return 0.0f;
  if (y >= 1.0f) return 23.5f;
  return 29.5f + 0.8f * fmaxf(0.0f, -__logf(fmaxf(y, 1.0e-8f) * 100.0f));
}

// e^z, |z| < 80, as 2^m (1 + p): 1 + p rounded, with what the rounding cut off
// in lo.  p = expm1(r), |r| <= ln2 / 2, by a polynomial fitted at Chebyshev
// points (1e-8 of e^r).
static __device__ __forceinline__ float core_exp(float z, int &m, float &lo) {
  const float g = fmaf(z, 1.44269504f, 12582912.0f), f = g - 12582912.0f;  // nearest integer (1.5 2^23 added)
  const float r = fmaf(f, 2.1219444e-4f, fmaf(f, -0.693359375f, z));  // ln2 = 0.693359375 - 2.12e-4
  float q = fmaf(1.39336521e-3f, r, 8.36318173e-3f);
  q = fmaf(q, r, 4.16664667e-2f);
  q = fmaf(q, r, 0.166665763f);
  q = fmaf(q, r, 0.5f);
  const float p = fmaf(r * r, q, r);
  const float e = 1.0f + p;
  lo = p - (e - 1.0f);
  m = __float_as_int(g) - 0x4B400000;
  return e;
}
static __device__ __forceinline__ float core_pow2(int m) { return __int_as_float((m + 127) << 23); }

static __device__ __forceinline__ float core_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// e^{-x^2}, with the rounding of x^2 made up for.  Below the normal range (x^2 from 87
// to 100, the far end of an undamped line's core) it is a subnormal number, not 0:
// the logarithms of the tables tell the two apart.
static __device__ __forceinline__ float core_gauss(float x, float x2) {
  if (x2 > 87.0f) return expf(-x2);
  int m;
  float lo;
  const float e = core_exp(-x2, m, lo);
  return fmaf(-fmaf(x, x, -x2), e, e) * core_pow2(m);
}

// c: 2^{4n} c_n, n = 1 .. 22, at c[n - 1] (16-byte aligned, 24 values).
static __device__ __forceinline__ float k916_inner(float x, float x2, float y, float A, float D, const float *c) {
  float cn[24];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const float4 v = reinterpret_cast<const float4 *>(c)[q];
    cn[4 * q] = v.x, cn[4 * q + 1] = v.y, cn[4 * q + 2] = v.z, cn[4 * q + 3] = v.w;
  }
  int m;
  float lo;
  const float e = core_exp(x, m, lo);
  const float r = core_rcp(e);
  const float X = e * core_pow2(m - 4), Y = r * core_pow2(-m - 4);
  float p = cn[CORE_TERMS - 1], n = cn[CORE_TERMS_NEG - 1];
#pragma unroll
  for (int t = CORE_TERMS - 2; t >= 0; --t) p = fmaf(p, X, cn[t]);
#pragma unroll
  for (int t = CORE_TERMS_NEG - 2; t >= 0; --t) n = fmaf(n, Y, cn[t]);
  p *= X;
  p = fmaf(p * (x + x), lo * r, p);
  // sin(xy) up to its sign: xy reduced by pi, an odd polynomial (8e-9)
  const float xy = x * y;
  const float f = fmaf(xy, 0.318309886f, 12582912.0f) - 12582912.0f;
  const float t = fmaf(f, -9.6765358e-4f, fmaf(f, -3.140625f, xy));
  const float t2 = t * t;
  float s = fmaf(2.60515162e-6f, t2, -1.98090405e-4f);
  s = fmaf(s, t2, 8.33305065e-3f);
  s = fmaf(s, t2, -0.166666582f);
  s = fmaf(s * t2, t, t);
  return core_gauss(x, x2) * (fmaf(s * s, D, A) + fmaf(n, Y, p));
}

// The 8-node Gauss-Hermite rule, its nodes +-t_j paired: with v = x^2 + (y^2 -
// t^2), a pair is (al v + be) / (v^2 + k), al = 2 w y / pi, be = 2 t^2 al, k = 4
// y^2 t^2; the four fractions over one reciprocal.  g[j] = {y^2 - t^2, al, be, k}.
static __device__ __forceinline__ float k916_outer(float x2, const float4 *g) {
  float n[4], q[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 G = g[j];
    const float v = x2 + G.x;
    q[j] = fmaf(v, v, G.w);
    n[j] = fmaf(G.y, v, G.z);
  }
  const float n01 = fmaf(n[0], q[1], n[1] * q[0]), q01 = q[0] * q[1];
  const float n23 = fmaf(n[2], q[3], n[3] * q[2]), q23 = q[2] * q[3];
  return fmaf(n01, q23, n23 * q01) * core_rcp(q01 * q23);
}

}  // namespace helk
