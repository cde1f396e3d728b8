// Red + black sweep of FP32 levels on regular box grids (mg_sweep.cu): one launch reads the
// neighbouring boxes (or periodic images) in place, needs no ghost cells, and writes a second
// array of the same layout.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "mg_host.hpp"

namespace gbmg {

// A field of the next coarser level, on a lattice of its own.
struct CoarseField {
  float* base;  // first valid cell
  int E[3], nb[3];
  int pitch, plane;
  long long bstride;
};

// What a sweep starts from: its source, zero (the source is not read), or the source plus the
// piecewise-constant prolongation of the coarser level's field.
enum { SWEEP_SOURCE = 0, SWEEP_ZERO = 1, SWEEP_PROLONG = 2 };

// One level of one solve in a sweep launch.  All boxes have extents E on a lattice anchored at
// the domain's low corner, stored in lattice order (x fastest) every bstride elements, without
// ghost cells; src, rhs and dst share that layout.  The domain's low corner is local (0,0,0).
struct SweepGrid {
  const float* src;
  const float* rhs;
  float* dst;
  long long bstride;  // elements from one box to the next
  int N[3], E[3], nb[3];
  int pitch, plane;
  int periodic;       // bit d: dimension d is periodic
  int par0;           // colour parity of the domain's low corner
  float mh2;          // -h^2
  CoarseField coarse; // the coarser level's field (SWEEP_PROLONG); base null: none
  // sweeps of fabs with ghost cells (launch_sweep_f32_fabs): the layouts of rhs and dst, which above
  // have the source's
  int rpitch, rplane, dpitch, dplane;
  long long rstride, dstride;
  // tiling, set by plan_sweep: S strips of 4 cells x TY rows x ZC planes per block, hx / hy
  // strips and rows read around it, nt tiles per dimension, first tile of this grid
  int S, TY, ZC, hx, hy;
  int nt[3];
  int tile_begin;
  int pad_;
};

// Boxes of one size on a lattice anchored at the domain's low corner, stored in lattice order (x
// fastest) at a constant stride; offsets in elements of the fab.
struct Lattice {
  int N[3], E[3], nb[3];
  int pitch, plane;
  long long bstride, first;  // from one box to the next; the first box's first valid cell
};
bool lattice_of(const BoxArray& ba, const FabLayout& lay, Lattice* out);

// Residual + restriction of such a level (mg_sweep.cu): crhs = mean of the 8 children's
// residuals, cphi = 0.  The coarse fields lie on a lattice of their own.
struct RestrictGrid {
  SweepGrid g;  // src = phi, rhs; geometry
  float mih2;   // -1 / h^2
  int ZC;       // fine planes of a tile (even)
  int tiles_xy, tile_begin;
  CoarseField crhs, cphi;
};
struct RestrictPlan {
  int tiles = 0;
};
RestrictPlan plan_restrict(std::vector<RestrictGrid>& grids);
cudaError_t launch_restrict_f32(const RestrictGrid* grids, int ngrids, const RestrictPlan& p, cudaStream_t s);

// Fills the geometry of a level (not the pointers and the tiling); false if the level cannot
// be swept this way: boxes of one size on a lattice in lattice order, x extents in whole strips
// of 4 cells, even y extent, even periodic extents, FP32 without ghosts.
bool sweep_geometry(const BoxArray& ba, const FabLayout& lay, const int periodic[3], double h,
                    SweepGrid* out);

struct SweepPlan {
  int tiles = 0, threads = 0;
};
// Chooses the tiling of the grids of one launch; the grids of `back`, the same levels swept the
// other way, take it too.
SweepPlan plan_sweep(std::vector<SweepGrid>& grids, std::vector<SweepGrid>& back);

// Levels of at least kSweepMinCells cells are swept whole; in a launch over several solves, if
// their levels hold kSweepMinCellsBatch cells together.  Smaller ones keep half-sweeps.  Measured
// on GB300 with 2^14 / 2^16 / 2^18 / 2^20 for both: the 64^3 mixed solve 1.195 / 1.220 / 1.215 /
// 1.262 ms, 128^3 2.04 / 2.10 / 2.10 / 2.16 ms (one launch for two also counts on small levels);
// 8 problems of 32^3 to 64^3 together 3.48 / 3.50 / 3.34 / 3.39 ms, 48 of up to 128^3 18.8 / 18.7 /
// 18.9 / 19.2 ms (a step's lists are tiled anew).
extern const long long kSweepMinCells, kSweepMinCellsBatch;

cudaError_t launch_sweep_f32(const SweepGrid* grids, int ngrids, const SweepPlan& p, int start,
                             cudaStream_t s);

// The same sweep on a caller's FP32 fabs with ghost cells (not read): phi and rhs on lattices of any
// alignment, dst of phi's boxes without ghosts.
bool sweep_fabs_geometry(const BoxArray& ba, const FabLayout& phi, const FabLayout& rhs,
                         const FabLayout& dst, const int periodic[3], double h, SweepGrid* out);
cudaError_t launch_sweep_f32_fabs(const SweepGrid* grid, const SweepPlan& p, int phi_ghosts, cudaStream_t s);

}  // namespace gbmg
