// k_wings.cu -- the FP32 form of the interpolated-wings route (wings.cuh):
// the far kernel (node sums of the coarser panels) and the near kernel (the
// finer panels, the point-by-point work near the line centres, the way down
// the tree and the flush).  The lines' Algorithm 916 cores are left to
// k_core_f32, whose sums the near kernel adds.
//
// Against the direct kernel (k_voigt_f32, every line at every point of its
// window), far + near: 1e5 lines, 3e6 points 702 -> 259 us (69 % of the issue
// slots in near, 55 % in far), 1e6 lines at 12 conditions 21.0 -> 6.3 ms, 1e7
// lines 21.3 -> 9.2 ms, with errors against 64 bits no larger.
// Both kernels are bound by instruction issue at the
// latency that their warps in flight hide: 64 registers (4 CTAs an SM, a few
// spilled words in the near kernel's way down the tree) beat 128 (2 CTAs) by
// 5-10 %.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "helk_internal.cuh"
#include "voigt_common.cuh"
#include "voigt_f32.cuh"
#include "wings.cuh"

namespace helk {

// --------------------------------------------------------------- geometry --
WingGeom wing_geometry(int64_t n, double half, int num_sms) {
  WingGeom g;
  memset(&g, 0, sizeof g);
  g.ngrid = (int)n;
  g.lvl0 = n < (int64_t)2 * num_sms * WG_WARPS * (WG_S0 << 2) ? 0 : 2;
  const double widest = std::min(2.0 * half + 1.0, (double)n);
  g.lmax = -1;
  for (int l = 0; l < WG_LEVELS; ++l) {
    const int64_t s = (int64_t)WG_S0 << l;
    g.npan[l] = (int)(n / s);
    if ((double)s <= widest) g.lmax = l;
  }
  g.nstage = 1;
  while (g.nstage < WG_STAGES && wing_level(g, g.nstage) <= g.lmax) ++g.nstage;
  int64_t slots = 0, map = 0, far = 0;
  for (int k = 0; k < g.nstage; ++k) {
    const int l0 = wing_level(g, k);
    const int64_t span = (int64_t)WG_S0 << (l0 + 3);
    g.groups[k] = (int)((n + span - 1) / span);
    // the candidates of a group are shared among enough CTAs to fill the GPU
    g.parts[k] = k == 0 ? 1
                        : (int)std::min<int64_t>(16, std::max<int64_t>(1, (4ll * num_sms + g.groups[k] - 1) /
                                                                              g.groups[k]));
    g.mapoff[k] = (int)map;
    map += g.groups[k];
    if (k > 0) {
      far += (int64_t)g.groups[k] * g.parts[k];
      for (int l = l0; l < l0 + 3 && l <= g.lmax; ++l) {
        g.foff[l] = slots;
        slots += (int64_t)g.npan[l] * g.parts[k];
      }
    }
  }
  g.fslots = slots;
  g.nmap = (int)map;
  g.farblk = (int)far;
  return g;
}

// One warp per group: its candidate lines, the contiguous range of the list
// whose reference index lies within the condition's largest window half-width
// of the group's points.
__global__ void k_wingmap(int64_t nlines, const double *__restrict__ ckey, WingGeom G, const int *__restrict__ list,
                          const CondStats *__restrict__ cst, int32_t *__restrict__ lo, int32_t *__restrict__ hi) {
  const int cond = list ? list[blockIdx.y] : blockIdx.y;
  const int m = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (m >= G.nmap) return;  // warp-uniform
  int k = 0;
  while (k + 1 < G.nstage && m >= G.mapoff[k + 1]) ++k;
  const int64_t span = (int64_t)WG_S0 << (wing_level(G, k) + 3);
  const int64_t A = (int64_t)(m - G.mapoff[k]) * span;
  const int64_t B = min(A + span, (int64_t)G.ngrid);
  const long long W = cst[cond].wmax;
  const int64_t o = (int64_t)cond * G.nmap + m;
  int64_t first = 0, last = 0;
  if (W >= 0) {
    first = warp_search(ckey, 0, nlines, (double)A - (double)W, false);
    last = warp_search(ckey, first, nlines, (double)(B - 1) + (double)W, true);
  }
  if ((threadIdx.x & 31) == 0) {
    lo[o] = (int32_t)first;
    hi[o] = (int32_t)last;
  }
}

cudaError_t launch_wingmap(helk_ctx *c, int n_cond, const int *list, const WingGeom &g) {
  dim3 grid((unsigned)((g.nmap + 7) / 8), n_cond);
  ++c->launches;
  k_wingmap<<<grid, 256, 0, c->stream>>>(c->nlines, c->ckey, g, list, c->cstats, c->tile_lo, c->tile_hi);
  return cudaGetLastError();
}

// -------------------------------------------------------------- FP32 form --
// 12 nodes, panels at least 3 half-widths from the poles: truncation below
// 2.3e-8 of the profile at the closest distance (half an ulp is 6e-8), and
// falling with the twelfth power of it.
constexpr int W32_P = 12;
constexpr int W32_PS = 16;  // floats a node-sum slot
constexpr float W32_ETA2 = 9.0f;
// cos((2 j + 1) pi / 24), j = 0 .. 11
__device__ constexpr float W32_T[W32_P] = {0.99144486f,  0.92387953f,  0.79335334f,  0.60876143f,
                                           0.38268343f,  0.13052619f,  -0.13052619f, -0.38268343f,
                                           -0.60876143f, -0.79335334f, -0.92387953f, -0.99144486f};

// A line as a group's CTA holds it, positions counted from the group's first
// point.  u(i) = (i - c) beta + nphi.  Both quadrature terms are one rational
// function of r2 = u^2 + a^2,
//   n / d,  d = r2 (r2 (k1 r2 + m3) + C),  n = r2 (c3 r2 + c45) + c2:
// GH3 (Gh3Line) has k1 = 1, m3 = -3, C = 9/4 + 6 a^2, c45 = -3/2 c3, c2 = c3 (4 a^2
// + 3/2); GH1 is k1 = m3 = c3 = c45 = 0, C = 1, c2 = P1.
struct __align__(16) WingLine {
  int c;
  float nphi, beta, a2;
  float P1, c3, g1, g3;   // GH1 from g1 points off the centre on, GH3 from `core` up to g3 (margins included)
  float core, ib;         // ib: 1 / beta
  int ilo, ihi;           // window, clamped to just outside the group
};
static_assert(sizeof(WingLine) == 48, "WingLine must be 48 bytes");
constexpr float WING_FAR = 3.0e38f;

// The offset of point i from the line's centre, in points: monotone in i and,
// from the integer difference, the same whatever the group.
__device__ __forceinline__ float wing_off(const WingLine &L, int i) {
  return fmaf(L.nphi, L.ib, (float)(i - L.c));
}

// Whether a line is taken on a panel of s points whose ends have the offsets dl
// <= dh: as GH1 beyond g1, as GH3 between `core` and g3 (the method's
// boundaries with a margin of 1.5 points and 1e-6, so that every point of the
// panel is on one side in the per-point arithmetic), and far enough from the
// poles (sqrt(3/2) Doppler units nearer for the 3-node rule).  A line taken on a
// panel is also taken, by this test, on every panel inside it: the ends decide
// by themselves, and the distance from the poles gains a factor 5/3.  So a
// group may drop what its own panel takes.
struct WingReach {
  float d1, d3;
  __device__ __forceinline__ WingReach(const WingLine &L, float s) {
    const float hw = 0.5f * s * L.beta;
    const float q = fmaf(W32_ETA2 * hw, hw, -L.a2);
    d1 = q > 0.0f ? __fsqrt_rn(q) * L.ib * 1.000001f : 0.0f;
    d3 = q > 0.0f ? fmaf(1.2248f, L.ib, d1) : 0.0f;  // (q <= 0: far enough wherever the centre lies)
  }
  __device__ __forceinline__ bool takes(const WingLine &L, float dl, float dh) const {
    const float near = fmaxf(dl, -dh), far = fmaxf(dh, -dl), d = 0.5f * fabsf(dl + dh);
    return (near >= L.g1 && d >= d1) || (near >= L.core && far <= L.g3 && d >= d3);
  }
};

__device__ __forceinline__ void wing_line(const LineRec32 &R, int64_t gbase, int gspan, WingLine &L) {
  L.c = R.c - (int)gbase;
  L.nphi = -R.phi_k;
  L.beta = R.beta;
  L.a2 = R.a2;
  L.ib = __frcp_rn(R.beta);
  const float x1 = __fsqrt_rn(fmaxf(1.0e6f - R.a2, 0.0f)) * L.ib;
  const float x3 = __fsqrt_rn(fmaxf(100.0f - R.a2, 0.0f)) * L.ib;
  const bool all1 = R.a2 >= 1.0e6f;
  L.g1 = all1 ? -WING_FAR : fmaf(x1, 1.000001f, 1.5f);
  L.g3 = all1 ? -WING_FAR : fmaf(x1, 0.999999f, -1.5f);
  L.core = R.a2 >= 100.0f ? -WING_FAR : fmaf(x3, 1.000001f, 1.5f);
  L.P1 = R.P1;
  L.c3 = 6.0f * R.P3;
  L.ilo = (int)max((int64_t)R.ilo - gbase, (int64_t)-1);
  L.ihi = (int)min((int64_t)R.ihi - gbase, (int64_t)gspan);
}

// A line's coefficients on one panel (centre m, s points).
struct WingTerm {
  float uc, hw, a2, k1, m3, C, c3, c45, c2;
  __device__ __forceinline__ void zero() {
    uc = a2 = C = 1.0f;
    hw = k1 = m3 = c3 = c45 = c2 = 0.0f;
  }
  __device__ __forceinline__ void set(const WingLine &L, float m, float s) {
    uc = fmaf(m - (float)L.c, L.beta, L.nphi);
    hw = 0.5f * s * L.beta;
    a2 = L.a2;
    const bool gh1 = fmaf(uc, uc, a2) >= 1.0e6f;  // the panel lies on one side
    k1 = gh1 ? 0.0f : 1.0f;
    m3 = gh1 ? 0.0f : -3.0f;
    C = gh1 ? 1.0f : fmaf(6.0f, a2, 2.25f);
    c3 = gh1 ? 0.0f : L.c3;
    c45 = -1.5f * c3;
    c2 = gh1 ? L.P1 : L.c3 * fmaf(4.0f, a2, 1.5f);
  }
  // acc + the term at the node t
  __device__ __forceinline__ float add(float t, float acc) const {
    const float u = fmaf(t, hw, uc);
    const float r2 = fmaf(u, u, a2);
    const float p = fmaf(r2, fmaf(k1, r2, m3), C);
    const float n = fmaf(r2, fmaf(c3, r2, c45), c2);
    return fmaf(n, fast_rcp(r2 * p), acc);
  }
};

// Masks of a batch by list: bit b of word w is line 32 w + b.
constexpr int WG_WORDS = WG_CAP / 32;

// Adds the lines of a list (every `step`-th word of its masks from `w0` on;
// bit b of word w is line 32 w + b, or idx[32 w + b]) to a panel's node sums f
// (Kahan-compensated, in shared memory).  M lines at a time, one a lane of each
// of 32 / M groups of lanes, which share the nodes: nodes 12 M / 32 (lane / M)
// on; nine FP32 instructions and one MUFU reciprocal a node.  M = 8 suits the
// lists of the near kernel (a handful to some tens of lines), M = 32 (every
// node on a lane, no repeated coefficients) the longer ones of the far kernel.
template <int M>
__device__ __forceinline__ void list_nodes(const WingLine *rec, const uint32_t *mask, const uint16_t *idx, int nwords,
                                           int w0, int step, uint16_t *q, int lane, const float *T, float m, float s,
                                           float2 *f) {
  constexpr int NPL = W32_P * M / 32;  // nodes a lane
  const int grp = lane / M, at = lane % M;
  float acc[NPL], tn[NPL];
#pragma unroll
  for (int j = 0; j < NPL; ++j) {
    acc[j] = 0.0f;
    tn[j] = M == 32 ? W32_T[j] : T[grp * NPL + j];
  }
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
      WingTerm W;
      W.zero();
      if (i + at < take) W.set(rec[q[i + at]], m, s);
#pragma unroll
      for (int j = 0; j < NPL; ++j) acc[j] = W.add(tn[j], acc[j]);
    }
    if (fin) break;
    n -= 32;
    const uint16_t e = q[32 + lane];
    __syncwarp();
    q[lane] = e;
    __syncwarp();
  }
  if (any) {
    // sums over the M lanes of a group
    float v = 0.0f;
#pragma unroll
    for (int j = 0; j < NPL; ++j) {
#pragma unroll
      for (int o = M / 2; o >= 1; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
      v = at == j ? acc[j] : v;
    }
    if (at < NPL) {
      float2 a = f[grp * NPL + at];
      kahan_add(a.x, a.y, v);
      f[grp * NPL + at] = a;
    }
  }
  __syncwarp();
}

// Lists of a batch: the group's panels of its three levels, and (near kernel)
// the lines that overlap a warp's panel and are not taken on it or coarser.
enum { LST_L0 = 0, LST_L1 = 8, LST_L2 = 12, LST_U = 14, LST_N = 22 };

struct WingSmem {
  WingLine rec[WG_CAP];
  uint32_t mask[LST_N][WG_WORDS];
  uint16_t q[WG_WARPS][64];
  int wcnt[WG_WARPS];
};

// The candidate lines [first, last) of a group, every `stride`-th run of
// WG_THREADS of them: those that overlap the group and are not taken at its
// own level or coarser (gok: whether that level is worked and the group lies on
// the grid in full) are compacted, in list order, into S.rec; a batch is then
// sorted into lists (n: levels worked above -1; UNRES: also LST_U) and
// `work(count)` called.  s: points of a warp's panel.
template <bool UNRES, typename Work>
__device__ __forceinline__ void wing_scan(WingSmem &S, const LineRec32 *__restrict__ rec, int64_t first, int64_t last,
                                          int64_t stride, int64_t gbase, int64_t s, bool gok, bool ok2, bool ok1,
                                          bool ok0, int ngrid, Work work) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t gend = min(gbase + 8 * s, (int64_t)ngrid) - 1;
  const int gspan = (int)min(8 * s, (int64_t)1 << 30);
  const int nfull = (int)((gend + 1 - gbase) / s);  // panels on the grid in full
  const float fs = (float)s;
  int total = 0;
  for (int64_t l0 = first; l0 < last; l0 += stride) {
    const int64_t l = l0 + tid;
    WingLine L;
    bool keep = false;
    if (l < last) {
      const LineRec32 &R = rec[l];
      // lines whose whole window is core are the core kernel's
      const float ul = fmaf((float)(R.ilo - R.c), R.beta, -R.phi_k), uh = fmaf((float)(R.ihi - R.c), R.beta, -R.phi_k);
      if (R.ilo <= gend && R.ihi >= gbase && R.ilo <= R.ihi &&
          fmaxf(fmaf(ul, ul, R.a2), fmaf(uh, uh, R.a2)) >= 100.0f) {
        wing_line(R, gbase, gspan, L);
        keep = true;
        if (gok && L.ilo <= 0 && L.ihi >= gspan - 1)
          keep = !WingReach(L, 8.0f * fs).takes(L, wing_off(L, 0), wing_off(L, gspan - 1));
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
    if (total > WG_CAP - WG_THREADS || (total > 0 && l0 + stride >= last)) {  // CTA-uniform; total <= WG_CAP
      for (int t = 32 * w; t < total; t += WG_THREADS) {
        const bool in = t + lane < total;
        const WingLine &M = S.rec[min(t + lane, total - 1)];
        uint32_t mine = 0;  // lane k keeps list k's mask
        bool k2[2], k1[4];
        const int ilo = M.ilo, ihi = M.ihi;
        const int is = (int)s;
        float dl[8], dh[8];  // offsets of the panels' ends
#pragma unroll
        for (int p = 0; p < 8; ++p) {
          dl[p] = wing_off(M, p * is);
          dh[p] = wing_off(M, (p + 1) * is - 1);
        }
        {
          const WingReach T(M, 4.0f * fs);
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            k2[p] = in && ok2 && 4 * p + 4 <= nfull && ilo <= 4 * p * is && ihi >= 4 * (p + 1) * is - 1 &&
                    T.takes(M, dl[4 * p], dh[4 * p + 3]);
            const uint32_t m = __ballot_sync(0xffffffffu, k2[p]);
            if (lane == LST_L2 + p) mine = m;
          }
        }
        {
          const WingReach T(M, 2.0f * fs);
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            k1[p] = in && ok1 && 2 * p + 2 <= nfull && ilo <= 2 * p * is && ihi >= 2 * (p + 1) * is - 1 &&
                    T.takes(M, dl[2 * p], dh[2 * p + 1]);
            const uint32_t m = __ballot_sync(0xffffffffu, k1[p] && !k2[p >> 1]);
            if (lane == LST_L1 + p) mine = m;
          }
        }
        {
          const WingReach T(M, fs);
#pragma unroll
          for (int p = 0; p < 8; ++p) {
            const bool up = k2[p >> 2] || k1[p >> 1];
            const bool k0 = in && !up && ok0 && p + 1 <= nfull && ilo <= p * is && ihi >= (p + 1) * is - 1 &&
                            T.takes(M, dl[p], dh[p]);
            uint32_t m = __ballot_sync(0xffffffffu, k0);
            if (lane == LST_L0 + p) mine = m;
            if (UNRES) {
              m = __ballot_sync(0xffffffffu, in && !up && !k0 && ilo <= (p + 1) * is - 1 && ihi >= p * is);
              if (lane == LST_U + p) mine = m;
            }
          }
        }
        if (lane < (UNRES ? LST_N : LST_U)) S.mask[lane][t >> 5] = mine;
      }
      __syncthreads();
      work(total);
      total = 0;
      __syncthreads();
    }
  }
}

// Node sums of levels wing_level(k) .. + 2, k >= 1: a CTA takes a part of a
// group's candidates; warp w owns panel 8 grp + w of the lowest level and
// shares the coarser ones.
__global__ void __launch_bounds__(WG_THREADS, 3)
    k_wing_far32(const LineRec32 *__restrict__ rec_all, int64_t nlines, const int32_t *__restrict__ lo_all,
                 const int32_t *__restrict__ hi_all, WingGeom G, const int *__restrict__ cond_order,
                 const CondStats *__restrict__ cst, float *__restrict__ F_all) {
  __shared__ WingSmem S;
  __shared__ float2 fs[WG_WARPS][3][W32_P];
  if (G.nstage < 2) return;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cond = cond_order[blockIdx.y];
  int k = G.nstage - 1, b = blockIdx.x;
  while (k > 1 && b >= G.groups[k] * G.parts[k]) b -= G.groups[k] * G.parts[k], --k;
  const int top = wing_top(G, cst[cond].wmax), l0 = wing_level(G, k);
  if (l0 > top) return;  // no window holds a panel of this stage
  const int grp = b / G.parts[k], part = b % G.parts[k];
  const int64_t s = (int64_t)WG_S0 << l0;  // < 2^31 (l0 <= lmax)
  const int64_t gbase = (int64_t)grp * 8 * s;
  const bool u1 = l0 + 1 <= top, u2 = l0 + 2 <= top;
  const bool gok = l0 + 3 <= top && gbase + 8 * s <= G.ngrid;
  const int64_t m = (int64_t)cond * G.nmap + G.mapoff[k] + grp;
  const int64_t first = lo_all[m] + (int64_t)part * WG_THREADS, last = hi_all[m];
  if (lane < W32_P)
    for (int v = 0; v < 3; ++v) fs[w][v][lane] = make_float2(0.0f, 0.0f);
  __syncwarp();
  wing_scan<false>(S, rec_all + (int64_t)cond * nlines, first, last, (int64_t)G.parts[k] * WG_THREADS, gbase, s, gok,
                   u2, u1, true, G.ngrid, [&](int total) {
                     const int nw = (total + 31) >> 5;
#pragma unroll 1
                     for (int v = 0; v < 3; ++v) {  // own panel, then a share of the coarser ones
                       const int wide = 1 << v, pan = w >> v;
                       const float sp = (float)(s * wide);
                       list_nodes<32>(S.rec, S.mask[(v == 0 ? LST_L0 : v == 1 ? LST_L1 : LST_L2) + pan], nullptr, nw,
                                      w & (wide - 1), wide, S.q[w], lane, nullptr, ((float)pan + 0.5f) * sp - 0.5f,
                                      sp, fs[w][v]);
                     }
                   });
  __syncthreads();
  float *F = F_all + (int64_t)cond * G.fslots * W32_PS;
  const int np = G.parts[k];
  auto val = [&](int ww, int v) { return lane < W32_P ? fs[ww][v][lane].x - fs[ww][v][lane].y : 0.0f; };
  if (lane < W32_PS) {
    const int64_t i0 = (int64_t)grp * 8 + w;
    if (i0 < G.npan[l0]) F[(G.foff[l0] + i0 * np + part) * W32_PS + lane] = val(w, 0);
    if (u1 && w < 4) {
      const int64_t i1 = (int64_t)grp * 4 + w;
      if (i1 < G.npan[l0 + 1])
        F[(G.foff[l0 + 1] + i1 * np + part) * W32_PS + lane] = val(2 * w, 1) + val(2 * w + 1, 1);
    }
    if (u2 && w < 2) {
      const int64_t i2 = (int64_t)grp * 2 + w;
      if (i2 < G.npan[l0 + 2])
        F[(G.foff[l0 + 2] + i2 * np + part) * W32_PS + lane] =
            (val(4 * w, 2) + val(4 * w + 1, 2)) + (val(4 * w + 2, 2) + val(4 * w + 3, 2));
    }
  }
}

// Interpolation tables: [side][k][16] of a child's nodes in its parent (side 0:
// the lower half), [k][32] of the leaf's points, the nodes.
constexpr int W32_TABM = 2 * W32_P * W32_PS;
constexpr int W32_TABT = W32_TABM + W32_P * WG_S0;

// The values at a panel's nodes: a common part (hi + lo) and deviations from
// it.  The polynomial of the deviations carries their smaller rounding down
// the tree.
struct __align__(16) WingVal {
  float dev[W32_P];
  float hi, lo, pad[2];
};

// Both children of a panel at once: lanes 0 .. 11 the nodes of the lower half,
// lanes 16 .. 27 those of the upper (M: the lane's row of its child's matrix),
// plus the children's own node sums f.  The side `side` (or both, side < 0) is
// written to out[0] / out[1] (out + side for one side).
__device__ __forceinline__ void wing_children(const float (&M)[W32_P], const WingVal &v, float f, int lane, int side,
                                              WingVal *out) {
  const float vh = v.hi, vl = v.lo;  // `out` may be v itself
  float r = 0.0f;
#pragma unroll
  for (int k = 0; k < W32_P; ++k) r = fmaf(M[k], v.dev[k], r);
  r += f;
  const float mid = __shfl_sync(0xffffffffu, r, (lane & 16) + W32_P / 2);
  const int j = lane & 15;
  if (side < 0 || (lane >> 4) == side) {
    WingVal &o = out[side < 0 ? lane >> 4 : 0];
    if (j < W32_P) o.dev[j] = r - mid;
    if (j == 15) {
      const float h = vh + mid, z = h - vh;
      o.hi = h;
      o.lo = vl + ((vh - (h - z)) + (mid - z));
    }
  }
  __syncwarp();
}

// Lists of a warp's own lines: its panel's halves and leaves, and point by point
// on the leaves (GH1 throughout, or per point).
enum { SUB_H = 0, SUB_L = 2, SUB_G1 = 6, SUB_D = 10, SUB_N = 14 };
// Leaf lists up to this length are run point by point: at one point a lane that
// costs a line no more than a short list's nodes (1e5 lines, 3e6 points: near
// 211 us, 428 us with every leaf list through nodes).
constexpr int W32_LEAF_MIN = 6;

// NL: leaves of a warp's panel, 4 or 1 (WingGeom::lvl0 2 or 0).
template <int NL>
__global__ void __launch_bounds__(WG_THREADS, 4)
    k_wing_near32(const LineRec32 *__restrict__ rec_all, int64_t nlines, const int32_t *__restrict__ lo_all,
                  const int32_t *__restrict__ hi_all, WingGeom G, const int *__restrict__ cond_order,
                  const CondStats *__restrict__ cst, const float *__restrict__ F_all,
                  const float *__restrict__ tab, const float *__restrict__ kcore_all, double weight, int accumulate,
                  double *__restrict__ kappa_all) {
  constexpr int s = NL * WG_S0;          // points of a warp's panel
  constexpr int NH = NL / 2;             // its halves
  constexpr int NV = NL == 1 ? 3 : 9;    // node sums of a warp: own panel, pair, quarter; halves; leaves
  __shared__ WingSmem S;
  __shared__ float2 fs[WG_WARPS][NV][W32_P];
  __shared__ uint16_t s_uq[WG_WARPS][WG_CAP];  // lines not taken on the warp's panel or coarser
  __shared__ uint32_t s_sub[WG_WARPS][SUB_N][WG_WORDS];
  __shared__ WingVal s_top;
  __shared__ float s_T[W32_P];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cond = cond_order[blockIdx.y];
  const int ngrid = G.ngrid;
  const int64_t gbase = (int64_t)blockIdx.x * 8 * s;
  const int top = wing_top(G, cst[cond].wmax);
  if (lane < W32_P)
    for (int v = 0; v < NV; ++v) fs[w][v][lane] = make_float2(0.0f, 0.0f);
  if (tid < W32_P) s_T[tid] = tab[W32_TABT + tid];
  __syncwarp();
  const int64_t p0 = gbase + w * s;
  float sum[NL], comp[NL];
#pragma unroll
  for (int k = 0; k < NL; ++k) sum[k] = comp[k] = 0.0f;
  uint16_t *q = S.q[w], *uq = s_uq[w];
  uint32_t *sub = s_sub[w][0];
  const int64_t m = (int64_t)cond * G.nmap + blockIdx.x;
  const int left = (int)min((int64_t)s, (int64_t)ngrid - p0);  // points of the panel on the grid
  const int base = w * s;                                      // the panel's first point in the group
  wing_scan<true>(
      S, rec_all + (int64_t)cond * nlines, lo_all[m], hi_all[m], WG_THREADS, gbase, s,
      top >= G.lvl0 + 3 && gbase + 8 * s <= ngrid, top >= G.lvl0 + 2, top >= G.lvl0 + 1, top >= G.lvl0, ngrid,
      [&](int total) {
        const int nw = (total + 31) >> 5;
        // lines not taken on the panel: its halves, its leaves, point by point
        int n = 0;
        for (int wd = 0; wd < nw; ++wd) {
          const uint32_t b = S.mask[LST_U + w][wd];
          if ((b >> lane) & 1u) uq[n + __popc(b & ((1u << lane) - 1u))] = (uint16_t)(32 * wd + lane);
          n += __popc(b);
        }
        __syncwarp();
        const int nu = (n + 31) >> 5;
        int nleaf[NL];
#pragma unroll
        for (int p = 0; p < NL; ++p) nleaf[p] = 0;
#pragma unroll 1
        for (int t = 0; t < nu; ++t) {
          const bool in = 32 * t + lane < n;
          const WingLine L = S.rec[uq[in ? 32 * t + lane : 0]];
          const int ilo = L.ilo - base, ihi = L.ihi - base;
          uint32_t mine = 0;  // lane k keeps list k's mask
          float dl[NL], dh[NL];
#pragma unroll
          for (int p = 0; p < NL; ++p) {
            dl[p] = wing_off(L, base + 32 * p);
            dh[p] = wing_off(L, base + 32 * p + 31);
          }
          const WingReach T1(L, 64.0f), T0(L, 32.0f);
          bool kh[2] = {false, false};
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            kh[h] = in && top >= 1 && 64 * (h + 1) <= left && ilo <= 64 * h && ihi >= 64 * h + 63 &&
                    T1.takes(L, dl[2 * h], dh[2 * h + 1]);
            const uint32_t m = __ballot_sync(0xffffffffu, kh[h]);
            if (lane == SUB_H + h) mine = m;
          }
#pragma unroll
          for (int p = 0; p < NL; ++p) {
            const bool rest = in && !kh[p >> 1];
            bool k0 = false;
            if (NL > 1) {
              k0 = rest && top >= 0 && 32 * (p + 1) <= left && ilo <= 32 * p && ihi >= 32 * p + 31 &&
                   T0.takes(L, dl[p], dh[p]);
              const uint32_t m = __ballot_sync(0xffffffffu, k0);
              if (lane == SUB_L + p) mine = m;
              nleaf[p] += __popc(m);
            }
            // point by point, unless every covered point is a core point;
            // GH1 throughout where the nearest covered point is
            const int lo = max(ilo, 32 * p), hi = min(ihi, 32 * p + 31);
            const float ul = fmaf((float)(base + lo - L.c), L.beta, L.nphi);
            const float uh = fmaf((float)(base + hi - L.c), L.beta, L.nphi);
            const float rl = fmaf(ul, ul, L.a2), rh = fmaf(uh, uh, L.a2);
            const bool d = rest && !k0 && lo <= hi && fmaxf(rl, rh) >= 100.0f;
            const bool g1 = d && fminf(rl, rh) >= 1.0e6f && (L.a2 >= 1.0e6f || (ul > 0.0f) == (uh > 0.0f));
            uint32_t m = __ballot_sync(0xffffffffu, g1);
            if (lane == SUB_G1 + p) mine = m;
            m = __ballot_sync(0xffffffffu, d && !g1);
            if (lane == SUB_D + p) mine = m;
          }
          if (lane < SUB_N) sub[lane * WG_WORDS + t] = mine;
        }
        __syncwarp();
        // the panels' node sums: own, pair, quarter (shared with the other
        // warps), halves, leaves
#pragma unroll 1
        for (int v = 0; v < NV; ++v) {
          if (v >= 5) {
            const int nl = v == 5 ? nleaf[0] : v == 6 ? nleaf[1 % NL] : v == 7 ? nleaf[2 % NL] : nleaf[3 % NL];
            if (nl <= W32_LEAF_MIN) continue;
          }
          const bool out = v < 3;
          const int wide = out ? 1 << v : 1, pan = w >> v;
          const float sp = out ? (float)(s * wide) : v < 5 ? 64.0f : 32.0f;
          const float mid = out ? ((float)pan + 0.5f) * sp - 0.5f
                                : (float)base + ((float)(v < 5 ? v - 3 : v - 5) + 0.5f) * sp - 0.5f;
          const uint32_t *mk = out ? S.mask[(v == 0 ? LST_L0 : v == 1 ? LST_L1 : LST_L2) + pan]
                                   : sub + (v < 5 ? SUB_H + v - 3 : SUB_L + v - 5) * WG_WORDS;
          list_nodes<8>(S.rec, mk, out ? nullptr : uq, out ? nw : nu, out ? w & (wide - 1) : 0, wide, q, lane, s_T, mid,
                        sp, fs[w][v]);
        }
#pragma unroll 1
        for (int p = 0; p < NL; ++p) {
          const int ip = base + 32 * p + lane;
          const bool few =
              NL > 1 && (p == 0 ? nleaf[0] : p == 1 ? nleaf[1 % NL] : p == 2 ? nleaf[2 % NL] : nleaf[3 % NL]) <= W32_LEAF_MIN;
#pragma unroll 1
          for (int t = 0; t < nu; ++t) {
            const uint32_t m1 = sub[(SUB_G1 + p) * WG_WORDS + t];
            const uint32_t md = sub[(SUB_D + p) * WG_WORDS + t] | (few ? sub[(SUB_L + p) * WG_WORDS + t] : 0u);
            if ((m1 | md) == 0) continue;
            // the word's lines in order: first those GH1 throughout
            const int n1 = __popc(m1), nd = __popc(md);
            const uint32_t lt = (1u << lane) - 1u;
            if ((m1 >> lane) & 1u) q[__popc(m1 & lt)] = uq[32 * t + lane];
            if ((md >> lane) & 1u) q[n1 + __popc(md & lt)] = uq[32 * t + lane];
            __syncwarp();
            float part = 0.0f;
#pragma unroll 2
            for (int i = 0; i < n1; ++i) {
              const WingLine &D = S.rec[q[i]];
              const float u = fmaf((float)(ip - D.c), D.beta, D.nphi);
              const float v = fmaf(D.P1, fast_rcp(fmaf(u, u, D.a2)), part);
              part = ip >= D.ilo && ip <= D.ihi ? v : part;
            }
            // core points (r2 < 100) are left to the core kernel
#pragma unroll 2
            for (int i = n1; i < n1 + nd; ++i) {
              const WingLine &D = S.rec[q[i]];
              const float a2 = D.a2, c3 = D.c3;
              const float u = fmaf((float)(ip - D.c), D.beta, D.nphi);
              const float r2 = fmaf(u, u, a2);
              const float pp = fmaf(r2, r2 - 3.0f, fmaf(6.0f, a2, 2.25f));
              const float nn = c3 * fmaf(r2, r2 - 1.5f, fmaf(4.0f, a2, 1.5f));
              const bool gh1 = r2 >= 1.0e6f;
              const float v = fmaf(gh1 ? D.P1 : nn, fast_rcp(gh1 ? r2 : r2 * pp), part);
              part = ip >= D.ilo && ip <= D.ihi && r2 >= 100.0f ? v : part;
            }
#pragma unroll
            for (int k = 0; k < NL; ++k)
              if (k == p) kahan_add(sum[k], comp[k], part);
            __syncwarp();
          }
        }
      });
  __syncthreads();  // the batch's shared memory is free
  WingVal *tv = reinterpret_cast<WingVal *>(S.rec) + w * 10;
  float M[W32_P];
  if (top >= 0) {
#pragma unroll
    for (int k = 0; k < W32_P; ++k) M[k] = tab[((lane >> 4) * W32_P + k) * W32_PS + (lane & 15)];
    if (w == 0) {
      // the values at the nodes of the group's own panel from the
      // coarser levels, coarsest first
      const float *F = F_all + (int64_t)cond * G.fslots * W32_PS;
      if (lane < 16) reinterpret_cast<float *>(&s_top)[lane] = 0.0f;
      __syncwarp();
      for (int l = top; l >= wing_level(G, 1); --l) {
        const int64_t p = gbase / ((int64_t)WG_S0 << l);
        if (p >= G.npan[l]) continue;  // not on the grid in full: nor is any coarser one
        const int np = G.parts[(l - G.lvl0) / 3];
        const float *Fp = F + (G.foff[l] + p * np) * W32_PS + (lane & 15);
        float f = 0.0f;
        for (int i = 0; i < np; ++i) f += Fp[i * W32_PS];
        wing_children(M, s_top, f, lane, (int)(p & 1), &s_top);
      }
    }
  }
  __syncthreads();
  if (p0 >= ngrid) return;
  if (top >= 0) {
    // down the tree: the quarter, the pair, the warp's panel, its halves, its leaves
    const int j = min(lane & 15, W32_P - 1), h4 = w & 4, h2 = w & 6, side = lane >> 4;
    auto val = [&](int ww, int v) { return fs[ww][v][j].x - fs[ww][v][j].y; };
#pragma unroll 1
    for (int t = 0; t < (NL == 1 ? 3 : 6); ++t) {
      const float f = t == 0 ? (val(h4, 2) + val(h4 + 1, 2)) + (val(h4 + 2, 2) + val(h4 + 3, 2))
                      : t == 1 ? val(h2, 1) + val(h2 + 1, 1)
                      : t == 2 ? val(w, 0)
                               : val(w, (t == 3 ? 3 + side : t == 4 ? 5 + side : 7 + side) % NV);
      // tv[0 .. 2]: quarter, pair, own; 3, 4: halves; 5 .. 8: leaves
      const WingVal &v = t == 0 ? s_top : tv[t - 1];
      wing_children(M, v, f, lane, t == 0 ? (w >> 2) & 1 : t == 1 ? (w >> 1) & 1 : t == 2 ? w & 1 : -1,
                    t < 3 ? tv + t : t == 3 ? tv + 3 : t == 4 ? tv + 5 : tv + 7);
    }
#pragma unroll
    for (int k = 0; k < W32_P; ++k) M[k] = tab[W32_TABM + k * WG_S0 + lane];
  }
  const int E = cst[cond].scale_exp;
  const bool core = cst[cond].core_w1 != 0, unit = weight == 1.0;
  const float *kcore = kcore_all + (int64_t)cond * ngrid;
  double *kappa = kappa_all + (int64_t)cond * ngrid;
#pragma unroll
  for (int p = 0; p < NL; ++p) {
    const int64_t i = p0 + 32 * p + lane;
    if (i < ngrid) {
      // the sums as an unevaluated pair (two-sums), then 2^E of it: for weight
      // 1 scaled on the integer pipe (exact), one FP64 addition rounds
      float hi = sum[p], lo = -comp[p];
      auto add = [&](float x) {
        const float t = hi + x, z = t - hi;
        lo += (hi - (t - z)) + (x - z);
        hi = t;
      };
      if (top >= 0) {
        const WingVal &v = tv[NL == 1 ? 2 : 5 + p];
        float far = 0.0f;
#pragma unroll
        for (int k = 0; k < W32_P; ++k) far = fmaf(M[k], v.dev[k], far);
        add(v.hi);
        add(far);
        lo += v.lo;
      }
      if (core) add(kcore[i]);
      const double v = unit ? scaled_to_double(hi, E) + scaled_to_double(lo, E)
                            : ldexp(weight, E) * ((double)hi + (double)lo);
      kappa[i] = accumulate ? kappa[i] + v : v;
    }
  }
}

// ----------------------------------------------------------------- launch --
// Lagrange basis of the nodes of [-1, 1] at x, in barycentric form.
static void lagrange(int P, const double *t, double x, double *out) {
  double den = 0.0;
  for (int j = 0; j < P; ++j) {
    const double w = ((j & 1) ? -1.0 : 1.0) * sin((2 * j + 1) * PI / (2 * P));
    if (x == t[j]) {
      for (int i = 0; i < P; ++i) out[i] = i == j ? 1.0 : 0.0;
      return;
    }
    out[j] = w / (x - t[j]);
    den += out[j];
  }
  for (int j = 0; j < P; ++j) out[j] /= den;
}

void wing_tables(int P, int PS, std::vector<double> &tab) {
  std::vector<double> t(P), r(P);
  for (int j = 0; j < P; ++j) t[j] = cos((2 * j + 1) * PI / (2 * P));
  tab.assign((size_t)2 * P * PS + (size_t)P * WG_S0 + P, 0.0);
  for (int j = 0; j < P; ++j) tab[(size_t)2 * P * PS + (size_t)P * WG_S0 + j] = t[j];
  for (int side = 0; side < 2; ++side)
    for (int j = 0; j < P; ++j) {
      lagrange(P, t.data(), (side ? 0.5 : -0.5) + 0.5 * t[j], r.data());
      for (int k = 0; k < P; ++k) tab[((size_t)side * P + k) * PS + j] = r[k];
    }
  for (int i = 0; i < WG_S0; ++i) {
    lagrange(P, t.data(), (2.0 * i + 1.0 - WG_S0) / WG_S0, r.data());
    for (int k = 0; k < P; ++k) tab[(size_t)2 * P * PS + (size_t)k * WG_S0 + i] = r[k];
  }
}

helk_status ensure_wing32(helk_ctx *c, int n_cond, const WingGeom &g) {
  helk_status st = ensure_buf(c, (void **)&c->wingF, &c->wingF_cap,
                              std::max<int64_t>(1, g.fslots) * n_cond * W32_PS * 4, "wing sums");
  if (st != HELK_OK || c->wing_tab32) return st;
  std::vector<double> tab;
  wing_tables(W32_P, W32_PS, tab);
  const std::vector<float> f(tab.begin(), tab.end());
  float *p = nullptr;
  st = cuda_check(c, cudaMalloc((void **)&p, f.size() * 4), "wing tables");
  if (st != HELK_OK) return st;
  // on the context's stream and waited for, so that every stream finds it complete
  st = cuda_check(c, cudaMemcpyAsync(p, f.data(), f.size() * 4, cudaMemcpyHostToDevice, c->stream), "wing tables");
  if (st == HELK_OK) st = cuda_check(c, cudaStreamSynchronize(c->stream), "wing tables");
  if (st == HELK_OK)
    c->wing_tab32 = p;
  else
    cudaFree(p);
  return st;
}

cudaError_t launch_wing_far32(helk_ctx *c, int n_cond, const WingGeom &g) {
  ++c->launches;
  // a grid without coarser levels launches one CTA that finds nothing to do
  k_wing_far32<<<dim3((unsigned)std::max(1, g.farblk), n_cond), WG_THREADS, 0, c->stream>>>(
      c->rec32, c->nlines, c->tile_lo, c->tile_hi, g, c->cond_order, c->cstats, (float *)c->wingF);
  return cudaGetLastError();
}

cudaError_t launch_wing_near32(helk_ctx *c, int n_cond, const WingGeom &g, const helk_opts &o, double *kappa) {
  ++c->launches;
  auto near = g.lvl0 == 2 ? k_wing_near32<4> : k_wing_near32<1>;
  near<<<dim3((unsigned)g.groups[0], n_cond), WG_THREADS, 0, c->stream>>>(
      c->rec32, c->nlines, c->tile_lo, c->tile_hi, g, c->cond_order, c->cstats, (const float *)c->wingF,
      c->wing_tab32, c->kcore, o.weight, o.accumulate, kappa);
  return cudaGetLastError();
}

}  // namespace helk
