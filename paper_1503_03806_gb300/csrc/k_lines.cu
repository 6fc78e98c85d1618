// k_lines.cu -- line-list kernels: validation, ordering by nu0, per-condition
// line preparation (Sec. 2.3-2.4) and the grid-tile -> line-range map.
//
// This translation unit is compiled with --fmad=false: the quantities that
// decide which grid points a line covers (window bounds) and which method
// evaluates a point (a, ku) must be the correctly rounded results of the
// operations written here, with no contraction into FMA.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "helk_internal.cuh"
#include "voigt_common.cuh"

namespace helk {

// -------------------------------------------------------- validation ---
// Doubles as unsigned integers of the same order.
__device__ __forceinline__ unsigned long long order_key(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return b >> 63 ? ~b : b | 0x8000000000000000ull;
}
// ListShape::at by a CTA's first threads.
__device__ __forceinline__ void list_cuts(int64_t n, const double *nu0, double *cuts) {
  if (threadIdx.x <= LIST_CUTS) cuts[threadIdx.x] = nu0[(n - 1) * threadIdx.x / LIST_CUTS];
}
// The high word of a double as an unsigned integer of the same order.
__device__ __forceinline__ unsigned order_key32(double v) {
  const int h = __double2hiint(v);
  return (unsigned)h ^ ((unsigned)(h >> 31) | 0x80000000u);
}
constexpr int VALIDATE_THREADS = 256;

// (of a list that is not ordered the cuts are taken again when it is)
__global__ void k_validate(int64_t n, const double *__restrict__ nu0, const double *__restrict__ S0,
                           const double *__restrict__ El, const double *__restrict__ gair,
                           const double *__restrict__ gself, const double *__restrict__ ncoll,
                           const double *__restrict__ delta, const double *__restrict__ lmass,
                           const double *__restrict__ lweight, UploadStats *st) {
  int bad = 0;
  if (blockIdx.x == 0) list_cuts(n, nu0, st->cuts);
  // order keys of high words (one operation a line and field: 1e7 ordered lines upload
  // in 437 us, with whole doubles in 470, without these in 443); of the least their
  // complements
  unsigned ga = 0, gs = 0, nmax = 0, nmin = 0, mmin = 0;
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n;
       l += (int64_t)gridDim.x * blockDim.x) {
    double v = nu0[l];
    bool ok = isfinite(v) && v > 0.0 && isfinite(S0[l]) && S0[l] >= 0.0 && isfinite(gair[l]) &&
              gair[l] >= 0.0;
    if (El) ok = ok && isfinite(El[l]);
    if (gself) ok = ok && isfinite(gself[l]) && gself[l] >= 0.0;
    if (ncoll) ok = ok && isfinite(ncoll[l]);
    if (delta) ok = ok && isfinite(delta[l]);
    if (lmass) ok = ok && isfinite(lmass[l]) && lmass[l] > 0.0;
    if (lweight) ok = ok && isfinite(lweight[l]) && lweight[l] >= 0.0;
    bad += !ok;
    ga = max(ga, order_key32(gair[l]));
    if (gself) gs = max(gs, order_key32(gself[l]));
    if (ncoll) {
      const unsigned k = order_key32(ncoll[l]);
      nmax = max(nmax, k);
      nmin = max(nmin, ~k);
    }
    if (lmass) mmin = max(mmin, ~order_key32(lmass[l]));
    if (l + 1 < n && nu0[l + 1] < v && *(volatile int *)&st->unsorted < SORT_RUNS) {
      const int q = atomicAdd(&st->unsorted, 1);
      if (q < SORT_RUNS) st->run_end[q] = (int)(l + 1);
    }
  }
  if (bad) atomicAdd(&st->bad_lines, bad);
  // (of a list with bad values these mean nothing: it is refused.)  Raised by the CTA,
  // the five at once: by every warp, one after the other, 2e5 ordered lines uploaded in
  // 87 us, 83 now.
  __shared__ unsigned top[5][VALIDATE_THREADS / 32];
  const unsigned own[5] = {ga, gs, nmax, nmin, mmin};
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const unsigned m = __reduce_max_sync(0xffffffffu, own[q]);
    if ((threadIdx.x & 31) == 0) top[q][threadIdx.x >> 5] = m;
  }
  __syncthreads();
  if (threadIdx.x < 5) {
    unsigned m = 0;
    for (int w = 0; w < VALIDATE_THREADS / 32; ++w) m = max(m, top[threadIdx.x][w]);
    atomicMax(&st->top[threadIdx.x], m);
  }
}

cudaError_t launch_validate_lines(helk_ctx *c, int64_t n) {
  if (n <= 0) return cudaSuccess;
  int blocks = (int)((n + 255) / 256);
  if (blocks > c->num_sms * 8) blocks = c->num_sms * 8;
  ++c->launches;
  k_validate<<<blocks, VALIDATE_THREADS, 0, c->stream>>>(n, c->nu0, c->S0, c->has_E ? c->El : nullptr, c->gair,
                                            c->has_gself ? c->gself : nullptr,
                                            c->has_ncoll ? c->ncoll : nullptr,
                                            c->has_delta ? c->delta : nullptr,
                                            c->has_mass ? c->lmass : nullptr,
                                            c->has_weight ? c->lweight : nullptr, c->upload);
  return cudaGetLastError();
}

// ------------------------------------------- stable LSD radix sort (pairs) --
// Keys: 64-bit, values: 32-bit.  One pass per 8-bit digit; each pass is
// upsweep (per-tile digit counts) -> exclusive scan -> downsweep (stable
// scatter: warps own consecutive sub-ranges, ranks inside a warp batch come
// from the digit's peer lanes).
constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_TILE = 4096;  // elements per block

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__global__ void __launch_bounds__(RS_THREADS) k_rs_upsweep(const unsigned long long *__restrict__ keys,
                                                           int64_t n, int shift, uint32_t *counts,
                                                           int nblk) {
  __shared__ uint32_t h[256];
  for (int d = threadIdx.x; d < 256; d += RS_THREADS) h[d] = 0;
  __syncthreads();
  int64_t b0 = (int64_t)blockIdx.x * RS_TILE;
  int64_t b1 = b0 + RS_TILE < n ? b0 + RS_TILE : n;
  for (int64_t e = b0 + threadIdx.x; e < b1; e += RS_THREADS)
    atomicAdd(&h[(keys[e] >> shift) & 0xFF], 1u);
  __syncthreads();
  for (int d = threadIdx.x; d < 256; d += RS_THREADS) counts[(int64_t)d * nblk + blockIdx.x] = h[d];
}

// Exclusive scan of m counts in place, one block of 1024 threads.
__global__ void __launch_bounds__(1024) k_rs_scan(uint32_t *counts, int64_t m) {
  __shared__ uint32_t wsum[32];
  int64_t per = (m + 1023) / 1024;
  int64_t s0 = threadIdx.x * per, s1 = s0 + per < m ? s0 + per : m;
  uint32_t s = 0;
  for (int64_t i = s0; i < s1; ++i) s += counts[i];
  // block exclusive scan of s
  uint32_t v = s;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  if (lane == 31) wsum[w] = v;
  __syncthreads();
  if (w == 0) {
    uint32_t x = wsum[lane];
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    wsum[lane] = x;
  }
  __syncthreads();
  uint32_t excl = v - s + (w > 0 ? wsum[w - 1] : 0u);
  for (int64_t i = s0; i < s1; ++i) {
    uint32_t t = counts[i];
    counts[i] = excl;
    excl += t;
  }
}

__global__ void __launch_bounds__(RS_THREADS) k_rs_downsweep(
    const unsigned long long *__restrict__ kin, const uint32_t *__restrict__ vin,
    unsigned long long *__restrict__ kout, uint32_t *__restrict__ vout, int64_t n, int shift,
    const uint32_t *__restrict__ counts, int nblk) {
  __shared__ uint32_t h[256 * RS_WARPS];  // [digit][warp]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < 256 * RS_WARPS; i += RS_THREADS) h[i] = 0;
  __syncthreads();
  int64_t b0 = (int64_t)blockIdx.x * RS_TILE;
  int64_t b1 = b0 + RS_TILE < n ? b0 + RS_TILE : n;
  const int per = RS_TILE / RS_WARPS;
  int64_t w0 = b0 + (int64_t)w * per, w1 = w0 + per < b1 ? w0 + per : b1;
  // per-warp digit counts
  for (int64_t e0 = w0; e0 < w1; e0 += 32) {
    int64_t e = e0 + lane;
    const bool valid = e < w1;
    uint32_t d = valid ? (uint32_t)((kin[e] >> shift) & 0xFF) : 0u;
    uint32_t peers = warp_digit_peers(d, valid);
    if (valid && (peers & lanemask_lt()) == 0) h[d * RS_WARPS + w] += __popc(peers);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < 256; d += RS_THREADS) {
    uint32_t run = counts[(int64_t)d * nblk + blockIdx.x];
    for (int ww = 0; ww < RS_WARPS; ++ww) {
      uint32_t t = h[d * RS_WARPS + ww];
      h[d * RS_WARPS + ww] = run;
      run += t;
    }
  }
  __syncthreads();
  for (int64_t e0 = w0; e0 < w1; e0 += 32) {
    int64_t e = e0 + lane;
    bool valid = e < w1;
    unsigned long long k = valid ? kin[e] : 0ull;
    uint32_t d = valid ? (uint32_t)((k >> shift) & 0xFF) : 0u;
    uint32_t peers = warp_digit_peers(d, valid);
    if (valid) {
      uint32_t pos = h[d * RS_WARPS + w] + __popc(peers & lanemask_lt());
      kout[pos] = k;
      vout[pos] = vin[e];
    }
    __syncwarp();
    if (valid && (peers & lanemask_lt()) == 0) h[d * RS_WARPS + w] += __popc(peers);
    __syncwarp();
  }
}

__global__ void k_line_keys(int64_t n, const double *__restrict__ nu0, unsigned long long *keys,
                            uint32_t *vals) {
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n;
       l += (int64_t)gridDim.x * blockDim.x) {
    double v = nu0[l];
    if (v == 0.0) v = 0.0;  // -0 -> +0
    keys[l] = order_key(v);
    vals[l] = (uint32_t)l;
  }
}

// The order of a list that is a few ordered runs (sort_runs.cuh).  2e5 lines in 4
// runs: 48 us, against 320 us for the radix passes.
__global__ void k_merge_runs(SortRuns R, const double *__restrict__ nu0, uint32_t *__restrict__ perm) {
  const int64_t n = R.end[R.n - 1];
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n; l += (int64_t)gridDim.x * blockDim.x)
    perm[merged_place(R, l, [=](int64_t i) { return nu0[i]; })] = (uint32_t)l;
}

// Up to four fields a launch: into the order of perm, and back to their places.
constexpr int GATHER_FIELDS = 4;
constexpr int64_t GATHER_BYTES = (int64_t)64 << 20;
struct GatherSet {
  int m;
  double *field[GATHER_FIELDS], *tmp[GATHER_FIELDS];
};
__global__ void k_gather(int64_t n, const uint32_t *__restrict__ perm, GatherSet G) {
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n;
       l += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t p = perm[l];
    for (int f = 0; f < G.m; ++f) G.tmp[f][l] = G.field[f][p];
  }
}
// cuts: NULL, or where the cuts of the ordered list's centres go (its field 0)
__global__ void k_gather_back(int64_t n, GatherSet G, double *cuts) {
  if (cuts && blockIdx.x == 0) list_cuts(n, G.tmp[0], cuts);
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n;
       l += (int64_t)gridDim.x * blockDim.x)
    for (int f = 0; f < G.m; ++f) G.field[f][l] = G.tmp[f][l];
}

// All fields into the order of perm, as many at a time as there are scratch arrays.
static cudaError_t reorder_fields(helk_ctx *c, int64_t n, const uint32_t *perm, double *const *tmp, int ntmp) {
  double *fields[9] = {c->nu0, c->S0, c->has_E ? c->El : nullptr, c->gair,
                       c->has_gself ? c->gself : nullptr, c->has_ncoll ? c->ncoll : nullptr,
                       c->has_delta ? c->delta : nullptr, c->has_mass ? c->lmass : nullptr,
                       c->has_weight ? c->lweight : nullptr};
  const int gb = (int)std::min<int64_t>((n + 255) / 256, (int64_t)c->num_sms * 16);
  GatherSet G{};
  for (int f = 0; f <= 9; ++f) {
    if (f < 9 && fields[f]) {
      G.field[G.m] = fields[f];
      G.tmp[G.m] = tmp[G.m];
      ++G.m;
    }
    if (G.m == ntmp || (f == 9 && G.m > 0)) {
      c->launches += 2;
      k_gather<<<gb, 256, 0, c->stream>>>(n, perm, G);
      // the cuts straight to the pinned copy of the statistics that the upload waits for
      k_gather_back<<<gb, 256, 0, c->stream>>>(n, G, G.field[0] == c->nu0 ? c->upload_host->cuts : nullptr);
      G.m = 0;
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_sort_lines(helk_ctx *c, int64_t n, int descents, const int *run_end) {
  if (n <= 1) return cudaSuccess;
  const int nblk = (int)((n + RS_TILE - 1) / RS_TILE);
  // scratch: 2 key arrays, 2 value arrays, counts, one double array
  int64_t need = 2 * n * 8 + 2 * n * 4 + (int64_t)256 * nblk * 4 + n * 8 + 64;
  const bool merge = merge_pays(n, descents + 1);
  if (merge) need = (int64_t)GATHER_FIELDS * n * 8 + n * 4;
  helk_status st = ensure_buf(c, &c->tmp, &c->tmp_cap, need, "line sort scratch");
  if (st != HELK_OK) return cudaErrorMemoryAllocation;
  char *p = (char *)c->tmp;
  int gb = (int)((n + 255) / 256);
  if (gb > c->num_sms * 16) gb = c->num_sms * 16;
  if (merge) {
    double *tmp[GATHER_FIELDS];
    for (int f = 0; f < GATHER_FIELDS; ++f, p += n * 8) tmp[f] = (double *)p;
    uint32_t *perm = (uint32_t *)p;
    SortRuns R{};
    R.n = descents + 1;
    for (int r = 0; r < descents; ++r) R.end[r] = run_end[r];
    std::sort(R.end, R.end + descents);
    R.end[descents] = (int)n;
    ++c->launches;
    k_merge_runs<<<gb, 256, 0, c->stream>>>(R, c->nu0, perm);
    return reorder_fields(c, n, perm, tmp, GATHER_FIELDS);
  }
  unsigned long long *ka = (unsigned long long *)p;  p += n * 8;
  unsigned long long *kb = (unsigned long long *)p;  p += n * 8;
  uint32_t *va = (uint32_t *)p;                      p += n * 4;
  uint32_t *vb = (uint32_t *)p;                      p += n * 4;
  uint32_t *counts = (uint32_t *)p;                  p += (int64_t)256 * nblk * 4;
  p = (char *)(((uintptr_t)p + 15) & ~(uintptr_t)15);
  double *dtmp = (double *)p;
  ++c->launches;
  k_line_keys<<<gb, 256, 0, c->stream>>>(n, c->nu0, ka, va);
  for (int pass = 0; pass < 8; ++pass) {
    int shift = pass * 8;
    ++c->launches;
    k_rs_upsweep<<<nblk, RS_THREADS, 0, c->stream>>>(ka, n, shift, counts, nblk);
    ++c->launches;
    k_rs_scan<<<1, 1024, 0, c->stream>>>(counts, (int64_t)256 * nblk);
    ++c->launches;
    k_rs_downsweep<<<nblk, RS_THREADS, 0, c->stream>>>(ka, va, kb, vb, n, shift, counts, nblk);
    unsigned long long *tk = ka; ka = kb; kb = tk;
    uint32_t *tv = va; va = vb; vb = tv;
  }
  double *const tmp[3] = {(double *)ka, (double *)kb, dtmp};  // the keys are done with
  // the fields that a launch reads in random order stay in the L2 cache together
  // (1e7 lines in no order: 7740 us three at a time, 7170 one at a time)
  const int fields = (int)std::min<int64_t>(3, std::max<int64_t>(1, GATHER_BYTES / (8 * n)));
  return reorder_fields(c, n, va, tmp, fields);
}

// ------------------------------------------------------- line preparation --
struct PrepArgs {
  double mass;
  int cut_kind;
  double cut_value, cut_cap;
  double nu_min, dnu, idnu;  // idnu = 1 / dnu
  int64_t ngrid;
};

// Per line and condition, in the operation order of the definitions:
//   nu0' = nu0 + delta P                                   (Sec. 2.3 shift)
//   S    = S0 (Q0/Q) e^{-c2E/T + c2E/T0} (1-e^{-c2 nu0/T})/(1-e^{-c2 nu0/T0})
//   S   *= abundance weight of the line's species          (Sec. 2.1)
//   Gamma_L = (T0/T)^n (g_air (P - P/2) + g_self P/2)      (Sec. 2.3)
//   Gamma_D = nu0' sqrt(2 ln2 k_B T / m) / c               (Sec. 2.3)
//   a = sqrt(ln2) Gamma_L / Gamma_D, ku = sqrt(ln2)/Gamma_D,
//   S' = S sqrt(ln2/pi) / Gamma_D, window from the cutoff   (Sec. 2.4)
// blockIdx.y is the condition; records of condition k start at k * n.
// r^2 >= R at grid index i, by the FP64 definition (each operation rounded)
__device__ __forceinline__ bool prep_beyond(const PrepArgs &A, double i, double nu0p, double ku, double a2, double R) {
  const double u = ((A.nu_min + i * A.dnu) - nu0p) * ku;
  return u * u + a2 >= R;
}

// The grid indices around a line's centre at which r^2 crosses R: the last one
// on the left with r^2 >= R (-1: none on the grid) and the first on the right (n:
// none).  r^2 is monotone on either side of the centre (cf: the index nearest to
// it, unclamped), so an estimate (w: the crossing's distance in steps) is moved
// until the definition holds; past a few steps by bisection.
__device__ __forceinline__ void prep_cross(const PrepArgs &A, double cf, double w, double nu0p, double ku, double a2,
                                           double R, int &left, int &right) {
  const double n = (double)A.ngrid;
  // left: the largest i in [-1, cf] with r^2 >= R (index -1 stands for "none")
  double hi = fmin(cf, n - 1.0), i = fmin(fmax(floor(cf - w), -1.0), hi);
  int step = 0;
  while (i >= 0.0 && step < 6 && !prep_beyond(A, i, nu0p, ku, a2, R)) i -= 1.0, ++step;
  while (i + 1.0 <= hi && step < 6 && prep_beyond(A, i + 1.0, nu0p, ku, a2, R)) i += 1.0, ++step;
  if (step >= 6) {
    double lo = -1.0;  // beyond at lo (or lo = -1), not beyond past hi
    while (lo < hi) {
      const double m = floor(0.5 * (lo + hi + 1.0));
      if (prep_beyond(A, m, nu0p, ku, a2, R)) lo = m;
      else hi = m - 1.0;
    }
    i = lo;
  }
  left = (int)fmax(i, -1.0);
  // right: the smallest i in [cf, n] with r^2 >= R (index n stands for "none")
  double lo = fmax(cf, 0.0);
  i = fmax(fmin(ceil(cf + w), n), lo);
  step = 0;
  while (i < n && step < 6 && !prep_beyond(A, i, nu0p, ku, a2, R)) i += 1.0, ++step;
  while (i - 1.0 >= lo && step < 6 && prep_beyond(A, i - 1.0, nu0p, ku, a2, R)) i -= 1.0, ++step;
  if (step >= 6) {
    double h = n;
    while (lo < h) {
      const double m = floor(0.5 * (lo + h));
      if (prep_beyond(A, m, nu0p, ku, a2, R)) h = m;
      else lo = m + 1.0;
    }
    i = h;
  }
  right = (int)fmin(i, n);
}

__global__ void k_lineprep(int64_t n, const double *__restrict__ nu0, const double *__restrict__ S0,
                           const double *__restrict__ El, const double *__restrict__ gair,
                           const double *__restrict__ gself, const double *__restrict__ ncoll,
                           const double *__restrict__ delta, const double *__restrict__ lmass,
                           const double *__restrict__ lweight, PrepArgs A,
                           const CondArgs *__restrict__ conds, CondArgs single,
                           LineRec64 *__restrict__ rec_all, double *__restrict__ ckey,
                           CondStats *cst_all, WingExt64 *__restrict__ ext_all,
                           int32_t *__restrict__ ckey32, int *__restrict__ core_blk_all, int nblk) {
  const int cond = blockIdx.y;
  const CondArgs C = conds ? conds[cond] : single;
  LineRec64 *rec = rec_all + (int64_t)cond * n;
  CondStats *cst = cst_all + cond;
  unsigned long long evals = 0;
  long long wmax = -1;
  unsigned long long spmax = 0;
  int cw1 = 0;
  const double vth = sqrt(2.0 * LN2 * KB * C.T / (A.mass * AMU)) / CLIGHT;
  const double tfac_half = sqrt(T0 / C.T);  // (T0/T)^n for the usual n = 1/2
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n;
       l += (int64_t)gridDim.x * blockDim.x) {
    const double v0 = nu0[l];
    const double dl = delta ? delta[l] : 0.0;
    const double ga = gair[l];
    const double gs = gself ? gself[l] : ga;
    const double nc = ncoll ? ncoll[l] : 0.5;
    double S = S0[l];
    const double nu0p = v0 + dl * C.P;
    if (El) {
      const double E = El[l];
      const double boltz = exp(-C2 * E / C.T + C2 * E / T0);
      const double stim = v0 > 0.0 ? expm1(-C2 * v0 / C.T) / expm1(-C2 * v0 / T0) : T0 / C.T;
      S = S * C.q_ratio * boltz * stim;
    }
    if (lweight) S = S * lweight[l];
    const double tfac = (nc == 0.5) ? tfac_half : pow(T0 / C.T, nc);
    const double pself = 0.5 * C.P;
    const double gL = tfac * (ga * (C.P - pself) + gs * pself);
    const double gD = nu0p * (lmass ? sqrt(2.0 * LN2 * KB * C.T / (lmass[l] * AMU)) / CLIGHT : vth);
    // divisions: a and k_u are the correctly rounded results the definition gives,
    // so every method choice matches it
    const double a = SQRTLN2 * gL / gD;
    const double ku = SQRTLN2 / gD;
    const double Sp = S * SQRTLN2PI / gD;
    double cut;
    if (A.cut_kind == HELK_CUT_ABS) cut = A.cut_value;
    else if (A.cut_kind == HELK_CUT_LORENTZ) cut = fmin(A.cut_value * gL, A.cut_cap);
    else cut = INFINITY;
    double lo, hi;
    if (A.cut_kind == HELK_CUT_NONE) {
      lo = 0.0;
      hi = (double)(A.ngrid - 1);
    } else {
      lo = ceil((nu0p - cut - A.nu_min) / A.dnu);
      hi = floor((nu0p + cut - A.nu_min) / A.dnu);
      if (lo < 0.0) lo = 0.0;
      if (hi > (double)(A.ngrid - 1)) hi = (double)(A.ngrid - 1);
      if (lo > (double)A.ngrid) lo = (double)A.ngrid;
      if (hi < -1.0) hi = -1.0;
    }
    LineRec64 r;
    r.nu0p = nu0p;
    r.ku = ku;
    r.a = a;
    r.a2 = a * a;
    r.Sp = Sp;
    r.ilo = (int32_t)lo;
    r.ihi = (int32_t)hi;
    // Algorithm 916 per-line factors (only reachable when a < 10)
    if (a < 10.0) {
      r.erfcx_a = erfcx(a);
      double s1 = 0.0;
      for (int k = 0; k < A916_S1_TERMS; ++k) {
        double nh = (double)(k + 1) * A916_H;
        s1 += A916_EXP_NH2[k] / (nh * nh + a * a);
      }
      r.sig1 = s1;
    } else {
      r.erfcx_a = 0.0;
      r.sig1 = 0.0;
    }
    rec[l] = r;
    // reference index of the unshifted centre: non-decreasing in list order
    double ck = floor((v0 - A.nu_min) / A.dnu);
    if (ck < -4.0e15) ck = -4.0e15;
    if (ck > 4.0e15) ck = 4.0e15;
    const int k32 = (int)min(max((long long)ck, -2147483647ll), 2147483647ll);
    if (cond == 0) ckey[l] = ck;
    if (cond == 0 && ckey32) ckey32[l] = k32;
    if (ext_all && C.wings) {
      WingExt64 x;
      const double idnu = 1.0 / A.dnu, pos = (nu0p - A.nu_min) * idnu;
      const double cf = rint(pos), cc = fmin(fmax(cf, 0.0), (double)(A.ngrid - 1));
      const float step = (float)(1.0 / (ku * A.dnu));  // a Doppler unit in grid steps
      x.c = (int)cc;
      x.frac = (float)(pos - cc);
      x.gamma = (float)a * step;
      x.node = 1.2248f * step;
      if (r.a2 >= R2_GH1) {
        x.g1l = x.g3l = INT_MAX;
        x.g1r = x.g3r = INT_MIN;
      } else {
        prep_cross(A, cf, (double)(sqrtf((float)(R2_GH1 - r.a2)) * step), nu0p, ku, r.a2, R2_GH1, x.g1l, x.g1r);
        if (r.a2 >= R2_GH3) {
          x.g3l = INT_MAX;
          x.g3r = INT_MIN;
        } else {
          prep_cross(A, cf, (double)(sqrtf((float)(R2_GH3 - r.a2)) * step), nu0p, ku, r.a2, R2_GH3, x.g3l, x.g3r);
        }
      }
      ext_all[(int64_t)cond * n + l] = x;
      // the core reach, as k_pack32 keeps it for the FP32 form
      const long long key = (long long)ck;
      const int clo = r.a2 >= R2_GH3 ? 1 : max(r.ilo, x.g3l + 1), chi = r.a2 >= R2_GH3 ? 0 : min(r.ihi, x.g3r - 1);
      int w1 = 0;
      if (clo <= chi) w1 = (int)min(max(key - clo, chi - key) + 1, 2000000000ll);
      cw1 = max(cw1, w1);
      const int blk = min(max(k32 >> 12, 0), nblk - 1);  // CORE_BLK_PTS = 2^12
      const unsigned peers = __match_any_sync(__activemask(), blk);
      const int wblk = __reduce_max_sync(peers, w1);
      if ((int)(threadIdx.x & 31) == __ffs(peers) - 1 && wblk > 0)
        atomicMax(&core_blk_all[(int64_t)cond * nblk + blk], wblk);
    }
    if (r.ihi >= r.ilo) {
      evals += (unsigned long long)(r.ihi - r.ilo + 1);
      long long c0 = (long long)ck;
      long long h1 = c0 - r.ilo, h2 = (long long)r.ihi - c0;
      long long hw = h1 > h2 ? h1 : h2;
      if (hw > wmax) wmax = hw;
      unsigned long long sb = (unsigned long long)__double_as_longlong(Sp);
      if (sb > spmax) spmax = sb;
    }
  }
  // warp-aggregate then one atomic per warp
  for (int o = 16; o > 0; o >>= 1) {
    evals += __shfl_down_sync(0xffffffffu, evals, o);
    long long w2 = __shfl_down_sync(0xffffffffu, wmax, o);
    if (w2 > wmax) wmax = w2;
    unsigned long long s2 = __shfl_down_sync(0xffffffffu, spmax, o);
    if (s2 > spmax) spmax = s2;
    cw1 = max(cw1, __shfl_down_sync(0xffffffffu, cw1, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (evals) atomicAdd(&cst->evals, evals);
    if (wmax >= 0) atomicMax(&cst->wmax, wmax);
    if (spmax) atomicMax(&cst->spmax_bits, spmax);
    if (cw1 > 0) atomicMax(&cst->core_w1, cw1);
  }
}

static int line_blocks(helk_ctx *c, int64_t n, int n_cond) {
  int64_t blocks = (n + 255) / 256;
  const int64_t cap = std::max<int64_t>(1, (int64_t)c->num_sms * 16 / std::max(1, n_cond));
  if (blocks > cap) blocks = cap;
  return (int)std::max<int64_t>(1, blocks);
}

cudaError_t launch_lineprep(helk_ctx *c, int n_cond, const CondArgs *single, double mass,
                            const helk_cutoff &cut, const helk_grid &g, bool wings) {
  const int64_t n = c->nlines;
  if (n <= 0) return cudaSuccess;
  PrepArgs A{mass, cut.kind, cut.value, cut.cap, g.nu_min, g.dnu, 1.0 / g.dnu, g.n};
  const CondArgs one = single ? *single : CondArgs{};
  dim3 grid(line_blocks(c, n, n_cond), n_cond);
  ++c->launches;
  k_lineprep<<<grid, 256, 0, c->stream>>>(
      n, c->nu0, c->S0, c->has_E ? c->El : nullptr, c->gair, c->has_gself ? c->gself : nullptr,
      c->has_ncoll ? c->ncoll : nullptr, c->has_delta ? c->delta : nullptr,
      c->has_mass ? c->lmass : nullptr, c->has_weight ? c->lweight : nullptr, A,
      single ? nullptr : c->cond_dev, one, c->rec64, c->ckey, c->cstats,
      wings ? c->ext64 : nullptr, wings ? c->ckey32 : nullptr, wings ? c->core_blk : nullptr, core_blocks(g.n));
  return cudaGetLastError();
}

// ----------------------------------------------------- FP32 line records --
// The FP32 form's records straight from the line list.  The FP64 unit (1/64 of the
// FP32 rate) bounds the preparation, so FP64 is kept for what decides the
// windows -- the shifted centre, Gamma_L, the cutoff bounds -- and the rest runs on
// FP32 (high, low) pairs: the strength with its two kinds of exponential
// (relative error ~1e-10) and k_u, a and their products (~1e-13), each rounded to
// FP32 once.  The divisions by the grid step are products by 1 / dnu where no
// integer lies within their rounding.  What is left is ~30 FP64 operations a line
// and condition, still the bound: 1e6 lines, 12 conditions take 0.85 ms and 0.21 ms
// to finish the records, against 3.5 + 0.6 ms with the FP64 form's records and a
// packing pass; 1e7 lines, one condition 0.70 + 0.21 against 3.0 + 0.5 ms.
struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 f2_norm(float h, float l) {
  const float s = h + l;
  return F2{s, l - (s - h)};
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  const float p = a.h * b.h;
  return f2_norm(p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p))));
}
__device__ __forceinline__ F2 f2_div(F2 a, F2 b) {
  const float r = __frcp_rn(b.h), q = a.h * r;
  const float rem = fmaf(-q, b.l, fmaf(-q, b.h, a.h) + a.l);
  return f2_norm(q, rem * r);
}
// v as a pair, from its bits (no FP64 instruction for 2^-70 < |v| < 2^127 and 0); a v
// past FP32's range as 2^100, far beyond what an exponential or a width takes, and
// finite, so that its products are
__device__ __forceinline__ F2 f2_of(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7FF) - 1023;
  if (e > -70 && e < 127) {
    const unsigned sign = hi & 0x80000000u;
    const float h = __uint_as_float(sign | (unsigned)(e + 127) << 23 | (hi & 0xFFFFFu) << 3 | lo >> 29);
    const float l = (float)(lo & 0x1FFFFFFFu) * __int_as_float((e - 52 + 127) << 23);
    return F2{h, sign ? -l : l};
  }
  if (e == -1023) return F2{0.0f, 0.0f};
  if (e >= 127) return F2{__uint_as_float((hi & 0x80000000u) | 0x71800000u), 0.0f};
  const float h = (float)v;
  return F2{h, (float)(v - (double)h)};
}
// v = (h + l) 2^e with 1 <= |h| < 2, from the bits (a normal v)
__device__ __forceinline__ F2 f2_mant(double v, int &e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  e = (int)((b >> 52) & 0x7FF) - 1023;
  const unsigned sign = (unsigned)(b >> 63) << 31;
  const float h = __uint_as_float(sign | 0x3F800000u | (unsigned)((b >> 29) & 0x7FFFFFu));
  const float l = (float)(unsigned)(b & 0x1FFFFFFFu) * 0x1p-52f;
  return f2_norm(h, sign ? -l : l);
}
__device__ __forceinline__ F2 prep_mant(double v, int &e) {  // also a subnormal v
  if (__double2hiint(v) >= 23 << 20) return f2_mant(v, e);
  const F2 r = f2_mant(v * 0x1p200, e);
  e -= 200;
  return r;
}
__device__ __forceinline__ float f_pow2(int e) {  // 2^e, clamped to the FP32 normal range
  return __int_as_float((min(max(e, -126), 127) + 127) << 23);
}

// 2^{j/32}, j = 0 .. 31
__device__ constexpr float PREP_POW[32][2] = {
    {0x1.0000000000000p+0f, 0x0.0p+0f}, {0x1.059b0e0000000p+0f, -0x1.9d4f520000000p-25f}, {0x1.0b55860000000p+0f, 0x1.9f31220000000p-25f},
    {0x1.11301e0000000p+0f, -0x1.fdb4960000000p-25f}, {0x1.172b840000000p+0f, -0x1.c157420000000p-27f}, {0x1.1d48740000000p+0f, -0x1.d2e8ca0000000p-25f},
    {0x1.2387a60000000p+0f, 0x1.ceac480000000p-25f}, {0x1.29e9e00000000p+0f, -0x1.5c04240000000p-25f}, {0x1.306fe00000000p+0f, 0x1.4636e20000000p-25f},
    {0x1.371a740000000p+0f, -0x1.18aac60000000p-25f}, {0x1.3dea640000000p+0f, 0x1.8246840000000p-25f}, {0x1.44e0860000000p+0f, 0x1.8624b40000000p-30f},
    {0x1.4bfdae0000000p+0f, -0x1.593abc0000000p-25f}, {0x1.5342b60000000p+0f, -0x1.2c56100000000p-25f}, {0x1.5ab07e0000000p+0f, -0x1.5bd5ec0000000p-27f},
    {0x1.6247ec0000000p+0f, -0x1.f8b5500000000p-25f}, {0x1.6a09e60000000p+0f, 0x1.9fcef40000000p-26f}, {0x1.71f75e0000000p+0f, 0x1.1d8bee0000000p-25f},
    {0x1.7a11480000000p+0f, -0x1.829fd00000000p-25f}, {0x1.82589a0000000p+0f, -0x1.accc7c0000000p-26f}, {0x1.8ace540000000p+0f, 0x1.15506e0000000p-27f},
    {0x1.93737c0000000p+0f, -0x1.e647440000000p-25f}, {0x1.9c49180000000p+0f, 0x1.51f8480000000p-27f}, {0x1.a5503c0000000p+0f, -0x1.b83b540000000p-25f},
    {0x1.ae89fa0000000p+0f, -0x1.a94b140000000p-26f}, {0x1.b7f7700000000p+0f, -0x1.a094380000000p-25f}, {0x1.c199be0000000p+0f, -0x1.3d56b20000000p-27f},
    {0x1.cb720e0000000p+0f, -0x1.8837cc0000000p-27f}, {0x1.d5818e0000000p+0f, -0x1.822dbc0000000p-27f}, {0x1.dfc9740000000p+0f, -0x1.908c940000000p-25f},
    {0x1.ea4afa0000000p+0f, 0x1.52486c0000000p-27f}, {0x1.f507660000000p+0f, -0x1.246eb00000000p-26f}};

// e^z as v 2^m, z a pair (clamped to +-80000: 2^m is then far out of range): z = (32 m + j) ln2 / 32 + r, |r| <= ln2 / 64,
// 2^{j/32} from the table and e^r - 1 by its Taylor polynomial to r^4 (1.3e-12).
// small: e^z - 1 itself where m = j = 0 (no cancellation), else v 2^m - 1.
__device__ __forceinline__ F2 prep_exp(F2 z, int &m, bool minus1) {
  if (fabsf(z.h) > 80000.0f) z = F2{copysignf(80000.0f, z.h), 0.0f};
  const float g = fmaf(z.h, 0x1.715476p+5f, 12582912.0f), n = g - 12582912.0f;
  const int k = __float_as_int(g) - 0x4B400000;
  const float p = n * 0x1.62e4300000000p-6f, pe = fmaf(n, 0x1.62e4300000000p-6f, -p);
  const F2 r = f2_norm(z.h - p, fmaf(-n, -0x1.05c6100000000p-34f, z.l - pe));
  const float q = r.h * r.h * fmaf(r.h, fmaf(r.h, 1.0f / 24.0f, 1.0f / 6.0f), 0.5f);
  const F2 e1 = f2_norm(r.h, fmaf(r.h, r.l, q) + r.l);  // e^r - 1
  m = k >> 5;
  if (minus1 && k == 0) return e1;
  const float th = PREP_POW[k & 31][0], tl = PREP_POW[k & 31][1];
  const F2 t = f2_mul(F2{th, tl}, e1);
  const float s = th + t.h;  // |t| < |th|
  F2 v = f2_norm(s, (t.h - (s - th)) + (tl + t.l));
  if (minus1) {  // z <= 0: m <= 0
    const float sc = m < -100 ? 0.0f : f_pow2(m);
    v = F2{v.h * sc, v.l * sc};
    const float d = v.h - 1.0f, bb = d - v.h;
    v = f2_norm(d, ((v.h - (d - bb)) + (-1.0f - bb)) + v.l);
    m = 0;
  }
  return v;
}

// q = v / dnu rounded up (UP) or down to an integer, clamped to [-2^30, 2^31 - 1]:
// from v (1 / dnu) where no integer lies within the rounding of that or of the
// division (2^-46 |q|; both err by < 2^-51 |q|), else by the division itself.
// Adding 1.5 2^52 leaves the nearest integer in the low word; comparisons are made
// on the high words, so the common path is a product and three additions.  Zero
// (a window that begins on the grid's first point) is an integer too, but has no
// exponent for that comparison: it has its own test.
constexpr double PREP_MAGIC = 6755399441055744.0;
__device__ __noinline__ int prep_index_div(double v, double dnu, bool up) {
  const double q = v / dnu;
  if (q <= -1073741824.0) return -1073741824;
  return (int)fmin(up ? ceil(q) : floor(q), 2147483647.0);
}
template <bool UP>
__device__ __forceinline__ int prep_index(double v, double dnu, double idnu) {
  const double q = v * idnu, t = q + PREP_MAGIC, d = q - (t - PREP_MAGIC);
  const int hq = __double2hiint(q) & 0x7FFFFFFF, hd = __double2hiint(d), r = __double2loint(t);
  const int ad = hd & 0x7FFFFFFF;
  if (hq >= 0x41D00000 || ad == 0 || hq - ad >= 46 << 20) return prep_index_div(v, dnu, UP);
  return UP ? r + (hd >= 0 ? 1 : 0) : r - (hd < 0 ? 1 : 0);
}

// The FP32 records with strengths as a mantissa in [1, 2) -- Sp, and P1 and P3 from
// it -- and its binary exponent in erfcx_a's place; sig1's place: the centre was
// clamped to the grid.  k_pack32 finishes them.
__global__ void __launch_bounds__(256)
    k_prep32(int64_t n, const double *__restrict__ nu0, const double *__restrict__ S0, const double *__restrict__ El,
             const double *__restrict__ gair, const double *__restrict__ gself, const double *__restrict__ ncoll,
             const double *__restrict__ delta, const double *__restrict__ lmass, const double *__restrict__ lweight,
             PrepArgs A, const CondArgs *__restrict__ conds, CondArgs single, LineRec32 *__restrict__ rec_all,
             double *__restrict__ ckey, CondStats *cst_all) {
  const int cond = blockIdx.y;
  const CondArgs C = conds ? conds[cond] : single;
  LineRec32 *rec = rec_all + (int64_t)cond * n;
  CondStats *cst = cst_all + cond;
  unsigned long long evals = 0;
  long long wmax = -1;
  unsigned long long spmax = 0;
  const double idnu = A.idnu, pself = 0.5 * C.P, pair_p = C.P - pself;
  const F2 kE = f2_of(C.kE), cT = f2_of(C.cT), cT0 = f2_of(C2 / T0), kc = f2_of(C.kc), dnu2 = f2_of(A.dnu);
  const F2 lnT = f2_of(C.lnT);
  int eq;
  const F2 qr = prep_mant(C.q_ratio, eq);
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n;
       l += (int64_t)gridDim.x * blockDim.x) {
    const double v0 = nu0[l], ga = gair[l];
    const double gs = gself ? gself[l] : ga;
    const double nc = ncoll ? ncoll[l] : 0.5;
    const double nu0p = delta ? v0 + delta[l] * C.P : v0;
    // Gamma_L: in FP64 where it decides the window, as k_lineprep rounds it
    const double gP = ga * pair_p + gs * pself;
    double gL = C.tfac * gP;
    F2 gL2;
    if (nc != 0.5 && A.cut_kind != HELK_CUT_LORENTZ) {
      int m;
      const F2 t = prep_exp(f2_mul(f2_of(nc), lnT), m, false);
      const float sc = f_pow2(m);
      gL2 = f2_mul(F2{t.h * sc, t.l * sc}, f2_of(gP));
    } else {
      if (nc != 0.5) gL = pow(T0 / C.T, nc) * gP;
      gL2 = f2_of(gL);
    }
    LineRec32 q;
    if (A.cut_kind == HELK_CUT_NONE) {
      q.ilo = 0;
      q.ihi = (int)(A.ngrid - 1);
    } else {
      const double cut = A.cut_kind == HELK_CUT_ABS ? A.cut_value : fmin(A.cut_value * gL, A.cut_cap);
      q.ilo = min(max(prep_index<true>(nu0p - cut - A.nu_min, A.dnu, idnu), 0), (int)A.ngrid);
      q.ihi = max(min(prep_index<false>(nu0p + cut - A.nu_min, A.dnu, idnu), (int)(A.ngrid - 1)), -1);
    }
    // k_u, a and the centre
    const F2 nup = f2_of(nu0p);
    F2 k = kc;  // sqrt(ln2) nu0' / Gamma_D, for this line's mass
    if (lmass) {
      const F2 mm = f2_of(lmass[l]);
      const float rs = rsqrtf(mm.h), s = mm.h * rs;
      k = f2_mul(k, f2_norm(s, 0.5f * rs * (fmaf(-s, s, mm.h) + mm.l)));
    }
    const F2 ku = f2_div(k, nup);
    const F2 a = f2_mul(gL2, ku);
    const F2 beta = f2_mul(dnu2, ku);
    q.beta = beta.h;
    q.a = a.h;
    q.a2 = fmaf(a.h, a.h, 2.0f * a.h * a.l);
    const double pos = (nu0p - A.nu_min) * idnu, pt = pos + PREP_MAGIC;
    double cf = pt - PREP_MAGIC;
    q.c = __double2loint(pt);
    const int hp = __double2hiint(pos);
    const bool big = (hp & 0x7FFFFFFF) >= 0x41DFFFFF;  // |pos| >= 2^31 - 1024: beyond any grid
    const bool below = big ? hp < 0 : q.c < 0, above = big ? hp >= 0 : q.c > A.ngrid - 1;
    if (below || above) {
      q.c = below ? 0 : (int)(A.ngrid - 1);
      cf = (double)q.c;
    }
    q.phi_k = f2_mul(f2_of(nu0p - (A.nu_min + cf * A.dnu)), ku).h;
    // S' = S ku / sqrt(pi), as a pair of order one times 2^e
    int e = 0;
    F2 S{0.0f, 0.0f};
    const double s0 = S0[l], wt = lweight ? lweight[l] : 1.0;
    if (__double_as_longlong(s0) > 0 && __double_as_longlong(wt) > 0) {
      int e1;
      S = prep_mant(s0, e);
      if (El) {
        const double E = El[l];
        const F2 vv = f2_of(v0);
        S = f2_mul(S, prep_exp(f2_mul(f2_of(E), kE), e1, false));
        e += e1 + eq;
        S = f2_mul(S, qr);
        const F2 x = f2_mul(vv, cT), y = f2_mul(vv, cT0);
        S = f2_mul(S, vv.h < 1e-12f  // the limit T0 / T, to 1e-14
                          ? f2_div(cT, cT0)
                          : f2_div(prep_exp(F2{-x.h, -x.l}, e1, true), prep_exp(F2{-y.h, -y.l}, e1, true)));
      }
      if (lweight) {
        S = f2_mul(S, prep_mant(wt, e1));
        e += e1;
      }
      S = f2_mul(f2_mul(S, ku), F2{0x1.20dd760000000p-1f, -0x1.f7ac920000000p-26f});
      // mantissa to [1, 2)
      const int ex = ((__float_as_int(S.h) >> 23) & 0xFF) - 127;
      const float sc = f_pow2(-ex);
      S = F2{S.h * sc, S.l * sc};
      e += ex;
    }
    q.Sp = S.h;
    const F2 Sa = f2_mul(S, a);
    q.P1 = f2_mul(Sa, F2{0x1.20dd760000000p-1f, -0x1.f7ac920000000p-26f}).h;
    q.P3 = f2_mul(Sa, F2{0x1.8127460000000p-4f, 0x1.606f3c0000000p-29f}).h;
    q.erfcx_a = __int_as_float(e);
    q.sig1 = below || above ? 1.0f : 0.0f;
    rec[l] = q;
    // reference index of the unshifted centre: non-decreasing in list order
    long long c0 = prep_index<false>(v0 - A.nu_min, A.dnu, idnu);
    if (c0 <= -1073741824 || c0 >= 2147483647) {
      double ck = floor((v0 - A.nu_min) / A.dnu);
      ck = fmin(fmax(ck, -4.0e15), 4.0e15);
      c0 = (long long)ck;
    }
    if (cond == 0) ckey[l] = (double)c0;
    if (q.ihi >= q.ilo) {
      evals += (unsigned long long)(q.ihi - q.ilo + 1);
      wmax = max(wmax, max(c0 - q.ilo, (long long)q.ihi - c0));
      // the bits of S' as a double (its largest gives the common scale)
      if (S.h > 0.0f && e > -1023 && e < 1024) {
        const unsigned long long sb =
            ((unsigned long long)(e + 1023) << 52) | ((unsigned long long)(__float_as_uint(S.h) & 0x7FFFFFu) << 29);
        spmax = max(spmax, sb);
      }
    }
  }
  // warp-aggregate then one atomic per warp
  for (int o = 16; o > 0; o >>= 1) {
    evals += __shfl_down_sync(0xffffffffu, evals, o);
    wmax = max(wmax, __shfl_down_sync(0xffffffffu, wmax, o));
    spmax = max(spmax, __shfl_down_sync(0xffffffffu, spmax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (evals) atomicAdd(&cst->evals, evals);
    if (wmax >= 0) atomicMax(&cst->wmax, wmax);
    if (spmax) atomicMax(&cst->spmax_bits, spmax);
  }
}

cudaError_t launch_prep32(helk_ctx *c, int n_cond, const CondArgs *single, double mass, const helk_cutoff &cut,
                          const helk_grid &g) {
  const int64_t n = c->nlines;
  if (n <= 0) return cudaSuccess;
  PrepArgs A{mass, cut.kind, cut.value, cut.cap, g.nu_min, g.dnu, 1.0 / g.dnu, g.n};
  const CondArgs one = single ? *single : CondArgs{};
  ++c->launches;
  k_prep32<<<dim3(line_blocks(c, n, n_cond), n_cond), 256, 0, c->stream>>>(
      n, c->nu0, c->S0, c->has_E ? c->El : nullptr, c->gair, c->has_gself ? c->gself : nullptr,
      c->has_ncoll ? c->ncoll : nullptr, c->has_delta ? c->delta : nullptr, c->has_mass ? c->lmass : nullptr,
      c->has_weight ? c->lweight : nullptr, A, single ? nullptr : c->cond_dev, one, c->rec32, c->ckey, c->cstats);
  return cudaGetLastError();
}

// The records finished: strengths scaled by 2^-E (E from the largest S' of the
// condition, so every scaled term is <= 1 and the FP32 range covers 38 decades
// below it; a power of two, so exact), the Algorithm 916 factors, the core range.
__global__ void k_pack32(int64_t n, int64_t ngrid, const double *__restrict__ ckey, CondStats *cst_all,
                         LineRec32 *__restrict__ r32_all, int2 *__restrict__ core_all, int32_t *__restrict__ ckey32,
                         int *err_flags, int *__restrict__ core_blk_all, int nblk) {
  const int cond = blockIdx.y;
  LineRec32 *r32 = r32_all + (int64_t)cond * n;
  CondStats *cst = cst_all + cond;
  const unsigned long long sb = cst->spmax_bits;
  const int E = sb ? (int)(sb >> 52) - 1022 : 0;  // ilogb + 1
  if (blockIdx.x == 0 && threadIdx.x == 0) cst->scale_exp = E;
  int cw1 = 0;
  for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < n;
       l += (int64_t)gridDim.x * blockDim.x) {
    const long long key = (long long)ckey[l];
    const int k32 = (int)min(max(key, -2147483647ll), 2147483647ll);
    if (cond == 0) ckey32[l] = k32;
    LineRec32 q = r32[l];
    const bool clamped = q.sig1 != 0.0f;
    {
      // 2^(e - E) in two factors: the first step stays normal
      const int d = min(max(__float_as_int(q.erfcx_a) - E, -250), 120);
      const float f1 = f_pow2(d / 2), f2 = f_pow2(d - d / 2);
      q.Sp = q.Sp * f1 * f2;
      q.P1 = q.P1 * f1 * f2;
      q.P3 = q.P3 * f1 * f2;
    }
    if (q.a < 10.0f) {  // Algorithm 916 per-line factors, in FP32
      q.erfcx_a = erfcxf(q.a);
      float s1 = 0.0f;
      for (int k = 0; k < A916_S1_TERMS; ++k) {
        const float nh = (float)(k + 1) * (float)A916_H;
        s1 += (float)A916_EXP_NH2[k] / (nh * nh + q.a2);
      }
      q.sig1 = s1;
    } else {
      q.erfcx_a = 0.0f;
      q.sig1 = 0.0f;
    }
    r32[l] = q;
    // The line's core in the FP32 arithmetic of the Voigt kernels: points with
    // fma(u, u, a^2) < 100, u = fma(i - c, beta, -phi), so |u| < 10.  With the
    // centre on the grid (|phi| <= beta/2) that needs |i - c| <= (10 + |phi|)/beta.
    // With a centre off the grid, c clamped to the nearer end, phi has the
    // sign of i - c, so |u| = |i - c| beta + |phi| and the core needs
    // |i - c| < (10 - |phi|)/beta: none once |phi| >= 10.  The farthest core
    // point from the reference index bounds the core kernel's candidate
    // search.
    int2 core = make_int2(1, 0);
    int line_w1 = 0;  // 1 + the line's core reach, 0: no core
    if (q.a2 < 100.0f && q.ihi >= q.ilo && q.beta > 0.0f) {
      const float reach = clamped ? 10.001f - fabsf(q.phi_k) : 10.001f + fabsf(q.phi_k);
      if (reach > 0.0f) {
        // an upper bound (FP32 quotient, rounding covered by the margin of 2)
        const float dmaxf = ceilf(reach / q.beta) + 2.0f;
        // Both Voigt kernels take i - c exactly in FP32 only within 2^24
        // points of c, so a core must end within 2^23 points (beta above
        // ~1.2e-6: a Doppler width below ~7e5 grid steps); else the call is
        // reported as unsupported by the FP32 form.
        if (dmaxf >= 8388608.0f) atomicOr(err_flags, ERRF_F32_RANGE);
        const long long dmax = (long long)fminf(dmaxf, 4.0e9f);
        const long long clo = max((long long)q.ilo, (long long)q.c - dmax);
        const long long chi = min((long long)q.ihi, (long long)q.c + dmax);
        if (clo <= chi) {
          const long long w = max(key - clo, chi - key);
          line_w1 = (int)min(w + 1, 2000000000ll);
          cw1 = max(cw1, line_w1);
          core = make_int2((int)clo, (int)chi);
        }
      }
    }
    core_all[(int64_t)cond * n + l] = core;
    // The reach of the lines whose reference index lies in each block of
    // CORE_BLK_PTS grid points (the core kernel's candidate window): the
    // list is ordered by the index, so the lanes of a warp mostly share a
    // block and one atomic per block and warp suffices.
    const int blk = min(max(k32 >> 12, 0), nblk - 1);  // CORE_BLK_PTS = 2^12
    const unsigned peers = __match_any_sync(__activemask(), blk);
    const int wblk = __reduce_max_sync(peers, line_w1);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1 && wblk > 0)
      atomicMax(&core_blk_all[(int64_t)cond * nblk + blk], wblk);
  }
  for (int o = 16; o > 0; o >>= 1) cw1 = max(cw1, __shfl_down_sync(0xffffffffu, cw1, o));
  if ((threadIdx.x & 31) == 0 && cw1 > 0) atomicMax(&cst->core_w1, cw1);
}

cudaError_t launch_pack32(helk_ctx *c, int n_cond, const helk_grid &g) {
  const int64_t n = c->nlines;
  if (n <= 0) return cudaSuccess;
  dim3 grid(line_blocks(c, n, n_cond), n_cond);
  ++c->launches;
  k_pack32<<<grid, 256, 0, c->stream>>>(n, g.n, c->ckey, c->cstats, c->rec32,
                                        c->core_rng, c->ckey32, &c->stats->err_flags, c->core_blk,
                                        core_blocks(g.n));
  return cudaGetLastError();
}

// --------------------------------------------------------------- tile map --
// Lines overlapping grid tile [A, B) have their reference index in
// [A - W, B - 1 + W], W = max half-width of any window of the condition: a
// contiguous range of the nu0-ordered list, found by two searches.  One warp
// per tile searches 32-ary: each step the lanes probe 32 evenly spaced keys
// and a ballot narrows the range 32-fold (5 dependent loads for 1e6 lines
// instead of 20 for a binary search).

__global__ void k_tilemap(int64_t nlines, const double *__restrict__ ckey, int64_t ngrid, int tile,
                          int64_t ntiles, const CondStats *__restrict__ cst, int32_t *tlo,
                          int32_t *thi) {
  const int cond = blockIdx.y;
  const int64_t t = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5);
  if (t >= ntiles) return;  // warp-uniform
  const int64_t o = (int64_t)cond * ntiles + t;
  const long long W = cst[cond].wmax;
  const int lane = threadIdx.x & 31;
  if (W < 0) {  // no line has a non-empty window
    if (lane == 0) tlo[o] = thi[o] = 0;
    return;
  }
  const double A = (double)(t * tile);
  const double B = (double)((t + 1) * tile < ngrid ? (t + 1) * tile : ngrid);
  const double klo = A - (double)W, khi = B - 1.0 + (double)W;
  const int64_t first = warp_search(ckey, 0, nlines, klo, false);  // first key >= klo
  const int64_t last = warp_search(ckey, first, nlines, khi, true); // first key > khi
  if (lane == 0) {
    tlo[o] = (int32_t)first;
    thi[o] = (int32_t)last;
  }
}

cudaError_t launch_tilemap(helk_ctx *c, int n_cond, const helk_grid &g, int tile, int64_t ntiles) {
  dim3 grid((unsigned)((ntiles + 7) / 8), n_cond);  // 8 warps, one tile each
  ++c->launches;
  k_tilemap<<<grid, 256, 0, c->stream>>>(c->nlines, c->ckey, g.n, tile, ntiles, c->cstats,
                                         c->tile_lo, c->tile_hi);
  return cudaGetLastError();
}

// ------------------------------------------------------- condition order --
// Largest evaluation count first, so the persistent Voigt kernel's last
// items are the cheapest (ties keep the input order).
__global__ void k_cond_order(int n_cond, const CondStats *__restrict__ cst, int *order) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  for (int i = 0; i < n_cond; ++i) {
    const unsigned long long e = cst[i].evals;
    int j = i;
    while (j > 0 && cst[order[j - 1]].evals < e) {
      order[j] = order[j - 1];
      --j;
    }
    order[j] = i;
  }
}

cudaError_t launch_cond_order(helk_ctx *c, int n_cond) {
  ++c->launches;
  k_cond_order<<<1, 32, 0, c->stream>>>(n_cond, c->cstats, c->cond_order);
  return cudaGetLastError();
}

}  // namespace helk
