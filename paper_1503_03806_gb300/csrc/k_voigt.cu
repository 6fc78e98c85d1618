// k_voigt.cu -- the FP32 form of the line-tiled Voigt opacity kernel, which takes
// every point of every window (narrow windows, few lines and counting calls; wings.cuh
// has the route of the others, which shares the core kernel) (Sec. 2.3-2.4): FP32 profile evaluation on records with strengths scaled by
// 2^-E, Kahan-compensated FP32 accumulation per point, the result converted
// to FP64 and rescaled at the flush; its Algorithm 916 cores in a separate
// kernel that runs beside it on a second stream; the table of kernel shapes
// the autotuner times; and the precision dispatch of the Voigt launch.
// Persistent CTAs; warp w of a tile owns 32 NSLOT consecutive grid points;
// the candidate lines of successive tiles stream through a shared-memory
// ring filled by 1-D bulk copies (see the pipeline below).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "helk_internal.cuh"
#include "voigt_common.cuh"
#include "voigt_core.cuh"
#include "voigt_f32.cuh"

namespace helk {

// Whether a core evaluation at (x, y) lies in a cell where the surrogate
// network was validated (features as in k_mlp.cu).
// The routing decision is split into a per-line part (the row of validated
// cells for y = a, or -1 when a is outside the network's range) and a
// per-point part (the column of x = |u|), both as in the network's features.
__device__ __forceinline__ int surr_row(const SurrQueue *sq, float y) {
  if (!sq || !(y >= 1.0e-4f && y < 10.0f)) return -1;
  const float f2 = 0.4f * (log10f(y) + 4.0f) - 1.0f;
  const int cy = min(max((int)((f2 + 1.0f) * 0.5f * sq->ny), 0), sq->ny - 1);
  return cy * sq->nx;
}

__device__ __forceinline__ bool surr_route(const SurrQueue *sq, int row, float x) {
  const float f1 = 2.0f * asinhf(x) * (float)(1.0 / ASINH_XCORE) - 1.0f;
  const int cx = min(max((int)((f1 + 1.0f) * 0.5f * sq->nx), 0), sq->nx - 1);
  const int cell = row + cx;
  return (sq->mask[cell >> 5] >> (cell & 31)) & 1u;
}

// One queue slot per calling lane: the lanes that arrive together take one
// atomicAdd for all of them (a single counter would otherwise see one atomic
// per routed evaluation).
__device__ __forceinline__ unsigned long long surr_reserve(SurrQueue *sq) {
  namespace cg = cooperative_groups;
  const cg::coalesced_group g = cg::coalesced_threads();
  unsigned long long base = 0;
  if (g.thread_rank() == 0) base = atomicAdd(&sq->count, (unsigned long long)g.size());
  return g.shfl(base, 0) + g.thread_rank();
}

// Appends one core evaluation (x^2 + y^2 < 100) to the surrogate's queue when
// its cell is validated (the queue's kernel adds it later); false when it has
// to be evaluated here.
__device__ __forceinline__ bool core_routed(float Sp, float a, float x, int i, int srow, SurrQueue *sq, int cond) {
  if (srow < 0 || !surr_route(sq, srow, x)) return false;
  const unsigned long long slot = surr_reserve(sq);
  if (slot >= sq->cap) return false;
  sq->idx[slot] = i;
  sq->cond[slot] = cond;
  sq->w[slot] = Sp;
  sq->x[slot] = x;
  sq->y[slot] = a;
  return true;
}

// ---- FP32 line pipeline: a ring of F32_STAGES chunks of candidate lines,
// filled by 1-D bulk copies that complete on the stage's mbarrier, with no
// CTA-wide barrier in the main loop.  Every warp consumes the chunk stream in
// order; the warp that finishes a chunk last (a shared-memory counter per
// stage) refills that stage with the chunk F32_STAGES further on, fetching
// the next (condition, tile) item from the global counter when the current
// one has no lines left.  So warps may drift apart by several chunks instead
// of meeting at a barrier after each one.  Each chunk carries a header (item,
// first line, count); an item without lines gets one empty chunk so that its
// tile is still written, and an exhausted item counter ends the stream with
// an empty chunk of item -1.
constexpr int F32_STAGES = 5;

struct ChunkHdr {
  int item, l0, cnt, pad;
};

struct F32Pipe {
  ChunkHdr hdr[F32_STAGES];
  unsigned long long full[F32_STAGES];
  int done[F32_STAGES];
  int pending[F32_STAGES];  // parity + 1 of a copy in flight into the stage, else 0
  int item, pos, end, exhausted;  // the issuer's place in the stream
};

// Publishes chunk `seq` of the stream into stage seq % F32_STAGES.  Called by
// one thread at a time (the initial fill, then the last consumer of the chunk
// that used the stage before).
template <int LCH>
__device__ void f32_issue(F32Pipe &P, LineRec32 (*sl)[LCH], unsigned long long seq, const LineRec32 *rec_all,
                          int64_t nlines, const int32_t *tlo_all, const int32_t *thi_all, int64_t ntiles,
                          const int *cond_order, int nitems, DevStats *st) {
  const int s = (int)(seq % F32_STAGES);
  const uint32_t mb = smem_addr(&P.full[s]);
  if (P.item < 0 || P.pos >= P.end) {  // the current item has no lines left: take the next one
    int item = -1;
    if (!P.exhausted) {
      item = (int)atomicAdd(&st->tile_counter, 1u);
      if (item >= nitems) item = -1;
    }
    if (item < 0) {
      P.exhausted = 1;
      P.hdr[s] = ChunkHdr{-1, 0, 0, 0};
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb) : "memory");
      return;
    }
    const int cond = cond_order[item / ntiles];
    const int64_t t = (int64_t)cond * ntiles + item % ntiles;
    P.item = item;
    P.pos = tlo_all[t];
    P.end = thi_all[t];
    if (P.pos >= P.end) {
      P.hdr[s] = ChunkHdr{item, P.pos, 0, 0};
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb) : "memory");
      return;
    }
  }
  const int cnt = min(LCH, P.end - P.pos);
  const int cond = cond_order[P.item / ntiles];
  P.hdr[s] = ChunkHdr{P.item, P.pos, cnt, 0};
  P.pending[s] = (int)((seq / F32_STAGES) & 1ull) + 1;
  // the stage's previous contents were read through the generic proxy
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tma_load_1d(smem_addr(&sl[s][0]), rec_all + (int64_t)cond * nlines + P.pos,
              (uint32_t)(cnt * sizeof(LineRec32)), mb);
  P.pos += cnt;
}

// After a failed wait: wait (bounded) for the copies still in flight, so that
// none lands in shared memory after the CTA has left.
__device__ void f32_drain(F32Pipe &P, int *flags) {
  for (int s = 0; s < F32_STAGES; ++s) {
    const int pend = *((volatile int *)&P.pending[s]);
    if (pend) mbar_wait_bounded(smem_addr(&P.full[s]), (uint32_t)(pend - 1), flags, WAIT_LIMIT_NS);
  }
}

// MINB resident CTAs per SM: 3 (<= 85 registers a thread) or 2.
template <int BLOCK, int NSLOT, int LCH, bool COUNT, int MINB>
__global__ void __launch_bounds__(BLOCK, MINB)
    k_voigt_f32(const LineRec32 *__restrict__ rec_all, int64_t nlines,
                const int32_t *__restrict__ tlo_all, const int32_t *__restrict__ thi_all,
                int64_t ntiles, const int *__restrict__ cond_order, int n_cond, int ngrid,
                double weight, int accumulate, double *__restrict__ kappa_all, CondStats *cst,
                DevStats *st, SurrQueue *sq) {
  // Warp w of the CTA owns the WSPAN consecutive points starting at
  // base + w WSPAN; lane l holds points base + w WSPAN + 32 k + l.  Method
  // classes are decided per (line, warp), so only the warps whose span holds
  // a method boundary or the line core take the per-point path.
  constexpr int NW = BLOCK / 32;
  constexpr int TILE = BLOCK * NSLOT;
  constexpr int WSPAN = 32 * NSLOT;
  constexpr int LPL = LCH / 32;  // lines of a chunk per lane in the class pass
  static_assert(LCH % 32 == 0 && LPL * 3 <= 32, "3 class bits per line in one word");
  __shared__ __align__(128) LineRec32 sl[F32_STAGES][LCH];
  __shared__ __align__(8) F32Pipe P;
  __shared__ WarpLine s_wl[NW][32];
  const int lane = threadIdx.x & 31;
  const int nitems = (int)(ntiles * n_cond);
  if (threadIdx.x == 0) {
    for (int s = 0; s < F32_STAGES; ++s) {
      mbar_init(smem_addr(&P.full[s]), 1);
      P.done[s] = 0;
      P.pending[s] = 0;
    }
    P.item = -1;
    P.pos = P.end = 0;
    P.exhausted = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (unsigned long long q = 0; q < F32_STAGES; ++q)
      f32_issue<LCH>(P, sl, q, rec_all, nlines, tlo_all, thi_all, ntiles, cond_order, nitems, st);

  // cur: the item being accumulated; -2 before the first chunk (-1 marks the
  // end of the stream, so a CTA that gets no item at all still sees a change)
  int cur = -2, wbase = 0;
  // No stream is longer than every item's chunks plus the end markers: a
  // longer one means a logic error, reported instead of looping.
  const uint32_t max_seq = (uint32_t)min(
      (unsigned long long)nitems * (unsigned long long)(nlines / LCH + 2) + 2 * F32_STAGES, 0x7FFFFFFFull);
  // Compensated accumulation: each point sums KAHAN_GROUP lines plainly
  // into part[k] (relative error <= 31 u, all terms positive) and Kahan-adds
  // the partial into (sum, comp); total relative error < 2e-6.
  float sum[NSLOT], comp[NSLOT], part[NSLOT];
  int ngroup = 0;
  unsigned long long cnt[4] = {0, 0, 0, 0};
  for (uint32_t seq = 0;; ++seq) {
    const int s = (int)(seq % F32_STAGES);
    if (seq > max_seq) {
      if (lane == 0) {
        atomicOr(&st->err_flags, ERRF_TIMEOUT);
        f32_drain(P, &st->err_flags);
      }
      return;
    }
    if (!mbar_wait_bounded(smem_addr(&P.full[s]), (seq / F32_STAGES) & 1u, &st->err_flags, WAIT_LIMIT_NS)) {
      if (lane == 0) f32_drain(P, &st->err_flags);
      return;
    }
    const ChunkHdr h = P.hdr[s];
    if (h.item != cur) {
      if (cur >= 0) {  // the previous tile is complete: write it
        const int cond = cond_order[cur / ntiles];
        double *kappa = kappa_all + (int64_t)cond * ngrid;
        const int E = cst[cond].scale_exp;
        const double scale = ldexp(weight, E);
        const bool unit = weight == 1.0;
#pragma unroll
        for (int k = 0; k < NSLOT; ++k) {
          kahan_add(sum[k], comp[k], part[k]);
          const int i = wbase + lane + 32 * k;
          if (i < ngrid) {
            // 2^E (sum - comp): for weight 1 the two scaled values are formed on
            // the integer pipe (exact) and one FP64 subtraction rounds, the
            // same result as scaling the FP64 difference
            const double v = unit ? scaled_to_double(sum[k], E) - scaled_to_double(comp[k], E)
                                  : scale * ((double)sum[k] - (double)comp[k]);
            kappa[i] = accumulate ? kappa[i] + v : v;
          }
        }
        if (COUNT) {
          for (int r = 0; r < 4; ++r) {
            unsigned long long v = cnt[r];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0 && v) atomicAdd(&cst[cond].region[r], v);
            cnt[r] = 0;
          }
        }
      }
      if (h.item < 0) return;  // end of the stream
      cur = h.item;
      wbase = (int)((cur % ntiles) * TILE) + (threadIdx.x >> 5) * WSPAN;
#pragma unroll
      for (int k = 0; k < NSLOT; ++k) {
        sum[k] = 0.0f;
        comp[k] = 0.0f;
        part[k] = 0.0f;
      }
      ngroup = 0;
    }
    if (lane == 0) P.pending[s] = 0;
    const LineRec32 *buf = sl[s];
    const int cnum = h.cnt;
    // The chunk in groups of 32 lines: lane l prepares line 32 m + l for this
    // warp (method class: the extreme r^2 over the warp's covered points
    // [lo, hi] decides it, r^2(d) being monotone on each side of the line
    // centre in the FP32 arithmetic of the evaluation loops), then the warp
    // runs through the group.
    WarpLine *wl = s_wl[threadIdx.x >> 5];
    for (int m0 = 0; m0 < cnum; m0 += 32) {
    int nk[NKIND];
    {
      const int j = m0 + lane;
      WarpLine r;
      r.kind = KIND_MISS;
      if (j < cnum) prepare_warp_line<NSLOT>(buf[j], wbase, r);
      order_warp_lines(r, lane, wl, nk);
    }
    __syncwarp();
    run_warp_lines<NSLOT, COUNT>(wl, nk, wbase, lane, ngroup, sum, comp, part, cnt);
    __syncwarp();  // the group's records are overwritten next
    }
    // release the stage; the last warp out refills it
    __syncwarp();
    if (lane == 0) {
      __threadfence_block();
      if (atomicAdd(&P.done[s], 1) == NW - 1) {
        P.done[s] = 0;
        __threadfence_block();
        f32_issue<LCH>(P, sl, seq + F32_STAGES, rec_all, nlines, tlo_all, thi_all, ntiles, cond_order, nitems,
                       st);
      }
    }
  }
}

// ------------------------------------------------- Algorithm 916 cores --
// The points of every line's core (fma(u, u, a^2) < 100 in the FP32
// arithmetic of the wing kernels, which skip exactly these points), one thread
// per grid point.  The candidate lines of a warp's 32 points are those whose
// reference index lies within the condition's core reach of them (found by
// the warp's own search); the lanes screen 32 of them at a time by their core
// ranges and prepare those that reach the warp, one a lane, in shared memory;
// the warp then takes them in list order (deterministic): it fills the line's
// table of series weights and Gauss-Hermite constants, and each lane whose
// point lies in the core adds S' K(|u|, a) by one of the two forms of
// voigt_core.cuh (or appends the point to the surrogate's queue when routed).
// The per-point sums go to kcore (every point written), so the kernel can run
// beside others; they are added into kappa rescaled like the main sums.
// Kahan-compensated: hundreds of cores can overlap at a point.
// Bound by instruction issue (81 % of the slots, ~150 a line and warp): 1e5 lines, 3e6
// points 129 us, 12 conditions of 1e6 lines 3.38 ms (141 us and 4.53 ms with a
// recurrence over the series terms of each point).
constexpr int CORE_BLOCK = 128;

struct __align__(16) CoreLine {
  float c, beta, nphi, a2;  // c: reference index from the warp's first point
  float y, A, D, Sp;
  float xc2;                // core_inner(y)
  int lo, hi, pad;          // core points
};

// A line whose profile is smooth on the warp's 32 points (all of them core points)
// is summed at 10 Chebyshev nodes of the block, three lines a pass, and the node
// sums are interpolated at the points once, at the end: 30 evaluations in place
// of 96.  Smooth: the block's half-width h = 16 beta <= 0.3, and 2 |x| h <= 1.5
// where e^{-x^2} can carry the profile (interpolation error 3e-8 of it, and the
// profile varies by less than e^1.5 from the block's middle), or the block so far
// out (x^2 >= 7 - ln y) that the wing carries it; 1.5e-7 of the profile at most.
// Grids with ~50 points or more to a Doppler half-width get there: 1e6 lines on 3e6
// points of dnu = 0.001, cores of ~1200 points: 4.91 -> 3.01 ms.  Where no line can
// (CORE_NODE_BETA), the kernel is compiled without: 48 registers in place of 71,
// 3.38 ms against 3.74 at 12 x 1e6 lines on 3e5 points of dnu = 0.1.
constexpr int CORE_NODES = 10, CORE_GROUPS = 3;
__device__ constexpr float CORE_NODE[CORE_NODES] = {0.987688341f, 0.891006524f, 0.707106781f, 0.4539905f, 0.156434465f, -0.156434465f, -0.4539905f, -0.707106781f, -0.891006524f, -0.987688341f};
__device__ constexpr float CORE_BARY[CORE_NODES] = {0.156434465f, -0.4539905f, 0.707106781f, -0.891006524f, 0.987688341f, -0.987688341f, 0.891006524f, -0.707106781f, 0.4539905f, -0.156434465f};

template <bool COUNT, bool NODES>
__global__ void __launch_bounds__(CORE_BLOCK)
    k_core_f32(const LineRec32 *__restrict__ rec_all, const int2 *__restrict__ core_all, int64_t nlines,
               const int32_t *__restrict__ ckey, int ngrid, float *__restrict__ kcore_all, CondStats *cst,
               SurrQueue *sq, const int *__restrict__ core_blk_all) {
  constexpr int NW = CORE_BLOCK / 32;
  __shared__ CoreLine s_line[NW][32];
  constexpr int NG = NODES ? CORE_GROUPS : 1;
  __shared__ __align__(16) float s_c[NW][NG][24];
  __shared__ float4 s_g[NW][NG][4];
  const int cond = blockIdx.y;
  const int cw1 = cst[cond].core_w1;
  if (cw1 == 0) return;  // no line of the condition has a core (its sums are not read)
  // each warp finds its own 32 points' candidate lines: no CTA barrier
  const int64_t A = (int64_t)blockIdx.x * CORE_BLOCK + (threadIdx.x & ~31);
  if (A >= ngrid) return;  // warp-uniform
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t B = min(A + 32, (int64_t)ngrid);
  // The candidate window: the condition's largest core reach, or, when that
  // is below a block, the largest reach of the lines whose reference index
  // lies in this block or its two neighbours (no line from a farther block
  // reaches the warp); the core reach grows with the line centre, so the
  // low-wavenumber warps scan far fewer lines.
  int64_t W = cw1 - 1;
  if (W < CORE_BLK_PTS - 32) {
    const int nblk = core_blocks(ngrid);
    const int b = (int)(A / CORE_BLK_PTS);
    const int *cb = core_blk_all + (int64_t)cond * nblk;
    int r = cb[b];
    if (b > 0) r = max(r, cb[b - 1]);
    if (b + 1 < nblk) r = max(r, cb[b + 1]);
    W = r - 1;  // -1: no line near this block has a core
  }
  // integer searches (FP64 is the scarce unit here)
  const int64_t first = warp_search(ckey, 0, nlines, A - W, false);
  const int64_t last = warp_search(ckey, first, nlines, B - 1 + W, true);
  const LineRec32 *rec = rec_all + (int64_t)cond * nlines;
  const int2 *core = core_all + (int64_t)cond * nlines;
  const int i = (int)(A + lane);
  // the lane's part of a line's tables: series term n = lane + 1, and the
  // Gauss-Hermite pair lane & 3
  float gauss = 0.0f;
  if (lane < CORE_TERMS) {
    const int n = lane + 1;
    gauss = n < A916_TERMS_F32 ? ldexpf(A916_GAUSS_F32[n], 4 * n) : A916_GAUSS_HIGH[n - A916_TERMS_F32];
    gauss *= 0.15915494f;  // h / pi
  }
  const float n2 = 0.25f * (float)((lane + 1) * (lane + 1));
  // nodes t^2 and weights 2 w / pi of the 8-node rule
  const int j = lane & 3;
  const float t2 = j == 0 ? 0.14530352f : j == 1 ? 1.33909729f : j == 2 ? 3.9269635f : 8.58863569f;
  const float w2 = j == 0 ? 0.420899261f : j == 1 ? 0.132291069f : j == 2 ? 1.08721817e-2f : 1.27071899e-4f;
  CoreLine *sl = s_line[wid];
  float(*sc)[24] = s_c[wid];
  float4(*sg)[4] = s_g[wid];
  const float flane = (float)lane;
  // the lane's node and group on the blocks taken through nodes (lanes 30, 31 idle)
  const int grp = lane / CORE_NODES;
  const float node = CORE_NODE[lane - CORE_NODES * grp];
  const float at = fmaf(16.0f, node, 15.5f);
  float F = 0.0f, Fc = 0.0f;
  bool nodes = false;
  float v = 0.0f, vc = 0.0f;
  unsigned long long n916 = 0, nterm = 0;
  for (int64_t l0 = first; l0 < last; l0 += 32) {
    const int64_t l = l0 + lane;
    int2 cr = make_int2(1, 0);
    if (l < last) cr = core[l];
    uint32_t todo = __ballot_sync(0xffffffffu, cr.x <= cr.y && cr.x < B && cr.y >= A);
    if (todo == 0) continue;
    __syncwarp();
    const bool mine = (todo >> lane) & 1u;
    bool smooth = false;
    CoreLine q;
    if (mine) {
      const LineRec32 L = rec[l];
      q.c = (float)(L.c - (int)A);  // within 2^23 points of a core point: exact
      q.beta = L.beta;
      q.nphi = -L.phi_k;
      q.a2 = L.a2;
      q.y = L.a;
      q.A = fmaf(-0.318309886f * L.a, L.sig1, L.erfcx_a);
      q.D = (L.a > 1.0e-15f ? __fdividef(0.318309886f, L.a) : 0.0f) - 2.0f * q.A;
      q.Sp = L.Sp;
      q.xc2 = core_inner(L.a);
      q.lo = cr.x;
      q.hi = cr.y;
      if (NODES && !sq && L.beta <= (float)CORE_NODE_BETA && cr.x <= A && cr.y >= A + 31 && A + 32 <= ngrid) {
        // every point is a core point when the two end points are (u is monotone)
        const float u0 = fmaf(0.0f - q.c, q.beta, q.nphi), u1 = fmaf(31.0f - q.c, q.beta, q.nphi);
        const float m0 = fminf(fabsf(u0), fabsf(u1)), m1 = fmaxf(fabsf(u0), fabsf(u1));
        smooth = fmaf(m1, m1, q.a2) < 100.0f &&
                 (m1 * q.beta <= 1.5f / 32.0f || (u0 * u1 > 0.0f && m0 * m0 >= 7.0f - __logf(fmaxf(q.y, 1.0e-30f))));
      }
    }
    // with nodes: the lines taken through them first, the others after them
    int slot = lane, nsm = 0;
    if (NODES) {
      const unsigned sm = __ballot_sync(0xffffffffu, smooth), lt = (1u << lane) - 1u;
      nsm = __popc(sm);
      slot = smooth ? __popc(sm & lt) : nsm + __popc(todo & ~sm & lt);
      todo = (unsigned)(((1ull << __popc(todo)) - 1ull) & ~((1ull << nsm) - 1ull));
    }
    if (mine) sl[slot] = q;
    __syncwarp();
    for (int s0 = 0; NODES && s0 < nsm; s0 += CORE_GROUPS) {
      nodes = true;
      const int li = min(s0 + grp, nsm - 1);
      const CoreLine &L = sl[li];
      const float u = fmaf(at - L.c, L.beta, L.nphi);
      const float x = fabsf(u), x2 = x * x, y = L.y, y2 = L.a2;
      const bool in = grp < CORE_GROUPS && s0 + grp < nsm;
      const bool inner = in && x2 < L.xc2;
      const unsigned bi = __ballot_sync(0xffffffffu, inner);
      const unsigned bo = __ballot_sync(0xffffffffu, in && !inner);
      if (bi && lane < CORE_TERMS) {
#pragma unroll
        for (int g = 0; g < CORE_GROUPS; ++g) {
          const CoreLine &G = sl[min(s0 + g, nsm - 1)];
          sc[g][lane] = gauss * G.y * core_rcp(n2 + G.a2);
        }
      }
      if (bo && lane < 4 * CORE_GROUPS) {
        const CoreLine &G = sl[min(s0 + (lane >> 2), nsm - 1)];
        const float al = w2 * G.y;
        sg[lane >> 2][j] = make_float4(G.a2 - t2, al, al * (t2 + t2), 4.0f * G.a2 * t2);
      }
      __syncwarp();
      float K = 0.0f;
      if (bi && inner) K = k916_inner(x, x2, y, L.A, L.D, sc[grp]);
      if (bo && in && !inner) {
        K = k916_outer(x2, sg[grp]);
        if (y < 1.0e-8f) K += core_gauss(x, x2);
      }
      if (in) kahan_add(F, Fc, L.Sp * K);
      __syncwarp();
    }
    for (; todo; todo &= todo - 1) {
      const CoreLine &L = sl[__ffs(todo) - 1];
      const float u = fmaf(flane - L.c, L.beta, L.nphi);
      const float y = L.y, y2 = L.a2, xc2 = L.xc2;
      bool in = i < ngrid && i >= L.lo && i <= L.hi && fmaf(u, u, y2) < 100.0f;
      const float x = fabsf(u), x2 = x * x;
      if (COUNT && in) {
        int n0, n1;
        a916_range_f32(x, n0, n1);
        ++n916;
        nterm += (unsigned long long)(n1 - n0 + 1);
      }
      if (sq && in) in = !core_routed(L.Sp, y, x, i, surr_row(sq, y), sq, cond);
      const bool inner = in && x2 < xc2;
      const unsigned bi = __ballot_sync(0xffffffffu, inner);
      const unsigned bo = __ballot_sync(0xffffffffu, in && !inner);
      if (bi) {
        if (lane < 24) sc[0][lane] = gauss * y * core_rcp(n2 + y2);
      }
      if (bo) {
        if (lane < 4) {
          const float al = w2 * y;
          sg[0][lane] = make_float4(y2 - t2, al, al * (t2 + t2), 4.0f * y2 * t2);
        }
      }
      __syncwarp();
      float K = 0.0f;
      if (bi && inner) K = k916_inner(x, x2, y, L.A, L.D, sc[0]);
      if (bo && in && !inner) {
        K = k916_outer(x2, sg[0]);
        if (y < 1.0e-8f) K += core_gauss(x, x2);
      }
      if (in) kahan_add(v, vc, L.Sp * K);
      __syncwarp();  // the tables are rebuilt for the next line
    }
  }
  float out = v - vc;
  if (NODES && nodes) {  // the node sums, interpolated at the points
    const float f = F - Fc;
    float num = 0.0f, den = 0.0f;
    const float xi = (flane - 15.5f) * (1.0f / 16.0f);
#pragma unroll
    for (int k = 0; k < CORE_NODES; ++k) {
      float fk = 0.0f;
#pragma unroll
      for (int g = 0; g < CORE_GROUPS; ++g) fk += __shfl_sync(0xffffffffu, f, CORE_NODES * g + k);
      const float r = __fdividef(CORE_BARY[k], xi - CORE_NODE[k]);
      num = fmaf(r, fk, num);
      den += r;
    }
    out += num / den;
  }
  if (i < ngrid) kcore_all[(int64_t)cond * ngrid + i] = out;
  if (COUNT) {
    for (int o = 16; o > 0; o >>= 1) {
      n916 += __shfl_down_sync(0xffffffffu, n916, o);
      nterm += __shfl_down_sync(0xffffffffu, nterm, o);
    }
    if (lane == 0 && n916) {
      atomicAdd(&cst[cond].region[0], n916);
      atomicAdd(&cst[cond].region[3], nterm);
    }
  }
}

// kappa += 2^E weight kcore at the points with a core sum (as k_voigt_f32's
// flush scales its sums); for weight 1 the scaled value is formed on the
// integer pipe, leaving one FP64 addition a point.
__global__ void __launch_bounds__(256)
    k_core_add(const float *__restrict__ kcore_all, int ngrid, double weight, double *__restrict__ kappa_all,
               const CondStats *cst) {
  const int cond = blockIdx.y;
  if (cst[cond].core_w1 == 0) return;
  const int E = cst[cond].scale_exp;
  const double scale = ldexp(weight, E);
  const bool unit = weight == 1.0;
  const float *kcore = kcore_all + (int64_t)cond * ngrid;
  double *kappa = kappa_all + (int64_t)cond * ngrid;
  // four points a thread per pass, their loads issued together
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < ngrid; i0 += 4 * stride) {
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t i = i0 + q * stride;
      v[q] = i < ngrid ? kcore[i] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t i = i0 + q * stride;
      if (v[q] != 0.0f) kappa[i] += unit ? scaled_to_double(v[q], E) : scale * (double)v[q];
    }
  }
}

cudaError_t launch_voigt_core(helk_ctx *c, int n_cond, const helk_grid &g, const helk_opts &o) {
  if (o.precision != HELK_PREC_F32_KAHAN || c->nlines <= 0) return cudaSuccess;
  SurrQueue *sq = o.surrogate ? c->squeue : nullptr;
  const dim3 grid((unsigned)((g.n + CORE_BLOCK - 1) / CORE_BLOCK), (unsigned)n_cond);
  ++c->launches;
  if (o.count_regions)
    k_core_f32<true, false><<<grid, CORE_BLOCK, 0, c->side_stream>>>(c->rec32, c->core_rng, c->nlines, c->ckey32,
                                                               (int)g.n, c->kcore, c->cstats, sq, c->core_blk);
  else if (c->core_nodes)
    k_core_f32<false, true><<<grid, CORE_BLOCK, 0, c->side_stream>>>(c->rec32, c->core_rng, c->nlines, c->ckey32,
                                                                     (int)g.n, c->kcore, c->cstats, sq, c->core_blk);
  else
    k_core_f32<false, false><<<grid, CORE_BLOCK, 0, c->side_stream>>>(c->rec32, c->core_rng, c->nlines, c->ckey32,
                                                                      (int)g.n, c->kcore, c->cstats, sq, c->core_blk);
  return cudaGetLastError();
}

cudaError_t launch_core_add(helk_ctx *c, int n_cond, const helk_grid &g, const helk_opts &o, double *kappa) {
  if (o.precision != HELK_PREC_F32_KAHAN || c->nlines <= 0) return cudaSuccess;
  const dim3 grid((unsigned)std::min<int64_t>((g.n + 255) / 256, (int64_t)c->num_sms * 8), (unsigned)n_cond);
  ++c->launches;
  k_core_add<<<grid, 256, 0, c->stream>>>(c->kcore, (int)g.n, o.weight, kappa, c->cstats);
  return cudaGetLastError();
}

// --------------------------------------------------------------- launch --
// FP32 kernel shapes, X(warps per CTA, slots per warp, candidate lines per
// pipeline stage, resident CTAs per SM the kernel is compiled for); a shape's
// code is its 1-based position in the list.  NSLOT is a template parameter
// (no per-slot bounds test in the hot loops) and the tile is 32 warps NSLOT
// points.  With 8 warps and 128-line stages the slots span 6..16, so that
// the number of tiles can be matched to whole waves of resident CTAs (equal
// tiles finish together, so a partial last wave idles the rest of the GPU);
// the other entries vary the CTA size (4, 12 warps) and the stage length (64,
// 256 lines, the latter also with 10-12 slots) for the autotuner.
#define HELK_F32_SHAPES(X)                                                                          \
  X(8, 6, 128, 3) X(8, 7, 128, 3) X(8, 8, 128, 3) X(8, 9, 128, 2) X(8, 10, 128, 2) X(8, 11, 128, 2)   \
  X(8, 12, 128, 2) X(8, 13, 128, 2) X(8, 14, 128, 2) X(8, 16, 128, 2) X(8, 8, 64, 3) X(8, 8, 256, 3)  \
  X(8, 7, 256, 3) X(4, 8, 128, 6) X(4, 9, 128, 4) X(12, 8, 128, 2) X(8, 10, 256, 2) X(8, 11, 256, 2)  \
  X(8, 12, 256, 2)
constexpr int F32_COUNT_CODE = 3;  // the counting variant (statistics): 8 warps, 8 slots, 128 lines
constexpr int F32_COUNT_NSLOT = 8, F32_COUNT_WARPS = 8, F32_COUNT_LCH = 128;

struct F32Shape {
  int warps, nslot, lch;
};
static const F32Shape kF32Shapes[] = {
#define X(W, NS, L, MB) {W, NS, L},
    HELK_F32_SHAPES(X)
#undef X
};
constexpr int F32_NSHAPES = (int)(sizeof(kF32Shapes) / sizeof(kF32Shapes[0]));

template <int W, int NS, int L, int MB>
static int f32_slots(helk_ctx *c) {
  return resident_ctas(c, k_voigt_f32<32 * W, NS, L, false, MB>, 32 * W);
}

bool voigt_shape_info(int precision, int code, int *points, int *warps, int *lines_per_stage) {
  if (precision != HELK_PREC_F32_KAHAN) return f64_shape_info(code, points, warps, lines_per_stage);
  if (code < 1 || code > F32_NSHAPES) return false;
  const F32Shape &s = kF32Shapes[code - 1];
  if (points) *points = 32 * s.warps * s.nslot;
  if (warps) *warps = s.warps;
  if (lines_per_stage) *lines_per_stage = s.lch;
  return true;
}

int voigt_shape_candidates(int precision, int *out, int max) {
  if (precision != HELK_PREC_F32_KAHAN) return f64_shape_candidates(out, max);
  int n = 0;
  for (int code = 1; code <= F32_NSHAPES && n < max; ++code) out[n++] = code;
  return n;
}

// Wave efficiency of ceil(n / tile) equal tiles on `slots` resident CTAs,
// times the share of a (line, warp) pair's work that is evaluation (the
// pair's fixed cost is about 2.5 slots).
static double f32_tile_score(int64_t n, int tile, int p, int slots) {
  const int64_t ntiles = (n + tile - 1) / tile;
  const double waves = (double)ntiles / slots;
  return waves / ceil(waves) * p / (p + 2.5);
}

int voigt_shape(helk_ctx *c, int precision, int count, int64_t n) {
  const int prec = precision == HELK_PREC_F32_KAHAN ? 1 : 0;
  if (!count && c->tuned_tile[prec] > 0 && c->tuned_n[prec] == n) return c->tuned_tile[prec];
  if (precision != HELK_PREC_F32_KAHAN) return f64_shape(c, count, n);
  if (count) return F32_COUNT_CODE;
  // without timing: the 8-warp, 128-line shapes by wave efficiency
  int best = F32_COUNT_CODE, code = 0;
  double best_score = -1.0;
#define X(W, NS, L, MB)                                                                  \
  ++code;                                                                                \
  if (W == 8 && L == 128) {                                                              \
    const double sc = f32_tile_score(n, 32 * W * NS, NS, f32_slots<W, NS, L, MB>(c));    \
    if (sc > best_score + 1e-9) {                                                        \
      best_score = sc;                                                                   \
      best = code;                                                                       \
    }                                                                                    \
  }
  HELK_F32_SHAPES(X)
#undef X
  return best;
}

cudaError_t launch_voigt(helk_ctx *c, int n_cond, const helk_grid &g, const helk_opts &o,
                         double *kappa, int shape, int64_t ntiles) {
  const int64_t nitems = ntiles * n_cond;
  if (o.precision != HELK_PREC_F32_KAHAN) return launch_voigt_f64(c, n_cond, g, o, kappa, shape, ntiles);
  SurrQueue *sq = o.surrogate ? c->squeue : nullptr;
  if (o.count_regions) {
    if (shape != F32_COUNT_CODE) return cudaErrorInvalidValue;
    constexpr int B = 32 * F32_COUNT_WARPS;
    auto kern = k_voigt_f32<B, F32_COUNT_NSLOT, F32_COUNT_LCH, true, 3>;
    ++c->launches;
    kern<<<persistent_grid(c, kern, B, nitems), B, 0, c->stream>>>(
        c->rec32, c->nlines, c->tile_lo, c->tile_hi, ntiles, c->cond_order, n_cond, (int)g.n, o.weight,
        o.accumulate, kappa, c->cstats, c->stats, sq);
    return cudaGetLastError();
  }
  int code = 0;
#define X(W, NS, L, MB)                                                                           \
  if (++code == shape) {                                                                          \
    auto kern = k_voigt_f32<32 * W, NS, L, false, MB>;                                             \
    ++c->launches;                                                                                 \
    kern<<<persistent_grid(c, kern, 32 * W, nitems), 32 * W, 0, c->stream>>>(                      \
        c->rec32, c->nlines, c->tile_lo, c->tile_hi, ntiles, c->cond_order, n_cond, (int)g.n,      \
        o.weight, o.accumulate, kappa, c->cstats, c->stats, sq);                                   \
    return cudaGetLastError();                                                                    \
  }
  HELK_F32_SHAPES(X)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace helk
