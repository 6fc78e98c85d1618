// wings.cuh -- geometry of the interpolated-wings route of the Voigt stage,
// shared by its FP32 and FP64 forms (k_wings.cu, k_wings64.cu).
//
// A line's profile is smooth away from its centre: on a panel of grid points
// that the line's window covers, on which one Gauss-Hermite method applies,
// and whose centre lies at least `eta` half-widths from the profile's poles
// (the line centre shifted by the quadrature nodes, +- i gamma), the profile
// is its polynomial interpolant through WG_P Chebyshev nodes of the panel to
// the arithmetic's resolution (the error falls as rho^-WG_P, rho = eta +
// sqrt(eta^2 - 1), the Bernstein ellipse through the poles).  So such a line
// costs WG_P evaluations on the panel, however many points it has, and the
// lines' values at the nodes are summed before anything is interpolated.
//
// Panels form a binary tree over the grid: level l has panels of WG_S0 2^l
// points.  A (line, panel) pair that passes the test above at level l and at
// no coarser one is taken there; a pair that passes at no level is evaluated
// point by point on the leaf (one point a lane).  Node sums are carried down
// the tree by the interpolation matrix of a child's nodes in its parent (exact
// for the polynomials, so no further truncation) and from the leaf's nodes to
// its points.  Only panels that lie on the grid in full exist, so every node is
// within the grid's range.
//
// A CTA works a group of 8 panels of one level, one a warp, and the two levels
// above it: the near kernel (stage 0) takes the panels of level lvl0, with the
// next two levels shared by its warps and any finer ones and the
// point-by-point work below; the far kernel (stage k >= 1) levels lvl0 + 3k and
// the next two.  A group scans its candidate lines once; lines taken at the
// group's own level (lvl0 + 3k + 3) or coarser are dropped at once.  lvl0 is 2
// (128 points a warp, 1024 a CTA), or 0 (32 and 256) on grids too short to give
// every SM two CTAs of the former.  Where the point-by-point kernels are taken instead:
// route.cuh.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "helk_internal.cuh"

namespace helk {

constexpr int WG_S0 = 32;                   // points of a leaf
constexpr int WG_LEVELS = 23;               // the coarsest panels have 2^27 points
constexpr int WG_STAGES = 7;
constexpr int WG_WARPS = 8;                 // panels (warps) a group
constexpr int WG_THREADS = 32 * WG_WARPS;
constexpr int WG_CAP = 480;                // lines of a batch in shared memory (32 * 15)

struct WingGeom {
  int ngrid;
  int lvl0;                     // level of the near kernel's panels (one a warp)
  int lmax;                     // coarsest level (-1: no panel of any level)
  int nstage;                   // stages with levels <= lmax (at least 1)
  int npan[WG_LEVELS];          // panels of a level that lie on the grid in full
  int64_t foff[WG_LEVELS];      // node-sum slots: first of a level (of the far stages)
  int64_t fslots;               // node-sum slots of a condition
  int groups[WG_STAGES];        // groups of a stage
  int parts[WG_STAGES];         // CTAs that share a group's candidate lines
  int mapoff[WG_STAGES];        // first entry of a stage in the candidate map
  int nmap;                     // candidate-map entries of a condition
  int farblk;                   // CTAs of the far kernel, coarsest stage first
};

// The lowest level of a stage's groups (one panel a warp).
__host__ __device__ inline int wing_level(const WingGeom &g, int stage) { return g.lvl0 + 3 * stage; }

// The coarsest level worth working for windows of at most wmax points on
// either side: a panel must lie inside a window.  Both kernels use it, so a
// level is either written by the far kernel and read by the near one, or
// neither.
__device__ __forceinline__ int wing_top(const WingGeom &g, long long wmax) {
  int l = g.lmax;
  while (l >= 0 && ((int64_t)WG_S0 << l) > 2 * wmax + 1) --l;
  return l;
}

// host: the geometry for a grid of n points, windows of at most
// `half` points on either side (a bound), on a GPU of num_sms SMs
WingGeom wing_geometry(int64_t n, double half, int num_sms);
// host: candidate line range of every group of every stage, for n_cond conditions:
// those in `list` (device), or all if it is NULL
cudaError_t launch_wingmap(helk_ctx *c, int n_cond, const int *list, const WingGeom &g);

// k_wings.cu: the FP32 form
helk_status ensure_wing32(helk_ctx *c, int n_cond, const WingGeom &g);
cudaError_t launch_wing_far32(helk_ctx *c, int n_cond, const WingGeom &g);
cudaError_t launch_wing_near32(helk_ctx *c, int n_cond, const WingGeom &g, const helk_opts &o, double *kappa);

// the interpolation tables for P nodes, rows padded to PS (FP64, on the host):
// [side][k][PS], [k][WG_S0], the nodes
void wing_tables(int P, int PS, std::vector<double> &tab);

// k_wings64.cu: the FP64 form (the far launch also takes the core sums)
helk_status ensure_wing64(helk_ctx *c, int n_cond, const WingGeom &g);
cudaError_t launch_wing_far64(helk_ctx *c, int n_cond, const int *list, const WingGeom &g, const helk_grid &grid);
cudaError_t launch_wing_near64(helk_ctx *c, int n_cond, const int *list, const WingGeom &g, const helk_grid &grid,
                               const helk_opts &o, double *kappa);

}  // namespace helk
