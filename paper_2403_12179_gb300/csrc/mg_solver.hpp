// Multigrid hierarchy shared by the single-solve driver (mg_solver.cu) and the batched /
// served drivers (mg_batch.cu).
#pragma once

#include "mg_runtime.hpp"
#include "mg_sweep.hpp"

namespace gbmg {

struct LevelData {
  std::shared_ptr<BoxArrayObj> bao;
  double h = 1.0;
  std::shared_ptr<FabObj> phi, rhs;
  OpTable smooth, rr, prolong, zero;
  // the stencil tables read neighbouring boxes directly (no ghost fill before them)
  bool direct = false;
  // sweeps ping-pong between phi and phi2 (same layout): fused (mg_fused.cu, ghost cells) or,
  // on FP32 levels over regular box grids, wide (mg_sweep.cu, neighbouring boxes read directly,
  // no ghost cells) -- where a launch covers enough cells, else the level's half-sweeps
  bool fused = false;
  bool wide = false;
  SweepGrid sweep_ab{}, sweep_ba{};  // phi -> phi2, phi2 -> phi (geometry and pointers)
  DevBufP sweep_dev;                 // both, tiled for a launch of their own
  bool wide_rr = false;              // its residual + restriction too (rr_grid)
  RestrictGrid rr_grid{};
  DevBufP rr_dev;
  RestrictPlan rr_plan{};
  SweepPlan sweep_plan{};            // no tiles: too small for a launch of its own
  // the first pre-smoothing sweep starts from zero without reading phi (nobody zeroes it), the first
  // post-smoothing sweep adds the prolongation (no kernel of its own): launches of their own sweep
  bool zero_start = false, add_start = false;
  long long cells() const { return bao->ba.dom.npts(); }
  std::shared_ptr<FabObj> phi2;
  FusedTable f_ab, f_ba;
};

struct Hierarchy {
  // cache key
  int64_t rhs_id = 0, phi_id = 0;
  int bc_key = 0;
  SolveParams p;
  mg_bc bc{};
  int dt = DT_F64;  // inner precision
  bool mixed = false;
  std::vector<LevelData> L;
  std::shared_ptr<FabObj> phi0, rhs0;  // the caller's fabs (FP64); staged: our own
  // An FP64 solve on its own over boxes not on a lattice works on one box of ours: phi and rhs are
  // copied there before the first cycle and phi back after the last, in place of a ghost fill before
  // every half-sweep of the finest level (GB300: 96 x 80 x 112 in boxes of 48, 2462 -> 2131 us; the three
  // copies and the last fill take 25 us).
  // Where the pool has no room for that the solve works on the caller's boxes, and tries again when
  // there is more room than there was (unstaged_room, of a hierarchy that is not staged for that reason).
  bool staged = false, unstaged = false;
  size_t unstaged_room = 0;
  OpTable stage_phi, stage_rhs, unstage_phi;
  std::shared_ptr<FabObj> r0;          // mixed: FP64 residual stored by each norm check (between the
                                       // scaling and that check, the second phi of the whole sweeps)
  bool direct0 = false;                // the norm check reads neighbouring boxes directly
  OpTable resid0, rhsabs0, scale0, correct0, zero0_64;
  DevBufP Mt, offr, offp, job;
  int N = 0;
  // levels [lc, L.size()) run as one coarse-cycle launch; lc == L.size(): not used
  int lc = 0;
  size_t csmem = 0;
  DevBufP cjob, coff;
  CoarseJob cjob_host{};
  // the same of a solve on its own, by a cluster of CTAs, from a finer level (slc <= lc; a batch, whose
  // jobs fill the SMs, takes one CTA a job; prepare_alone)
  int slc = 0, sranks = 1;
  size_t scsmem = 0;
  DevBufP scjob, scoff;
  bool alone = false;  // prepare_alone has run
  DevBufP dnorm;  // [0] residual norm bits, [1] rhs norm bits
  unsigned long long* hnorm = nullptr;
  BottomJob job_host{};
  bool job_shared = false;  // (a bottom level of the caller's fabs that share memory)
  // FP64 solves whose finest level starts each V-cycle with a red half-sweep: that
  // half-sweep of the next cycle also takes the red cells' residual norm of the current
  // iterate (it computes the same neighbour sums), replacing a separate residual pass; it
  // runs speculatively at the end of each step, saving the red values it replaces in save0
  // (null when the solve does not speculate), and is undone if the stop test ends the solve.
  // res0 holds, within each V-cycle, the black cells' residuals that the last pre-smoothing
  // half-sweep stores for the residual + restriction (stored0: level 0's residual +
  // restriction table reads them; store0 is that half-sweep's table).  Both are one-colour
  // arrays (half a row per row, see launch_rbgs_half).
  DevBufP save0, res0;
  OpTable store0;
  bool stored0 = false;
  // step graphs: [0] plain step, [1] first step of a speculating solve (a whole V-cycle,
  // then the next one's red half-sweep), [2] later steps (the V-cycle without that red
  // half-sweep, then the next one's)
  cudaGraphExec_t step_graph[3] = {nullptr, nullptr, nullptr};
  long long graph_kernels[3] = {0, 0, 0};
  cudaStream_t graph_stream = nullptr;
  bool graph_timed = false;                  // the step graphs record sweep_ev
  cudaEvent_t sweep_ev[2] = {nullptr, nullptr};
  ~Hierarchy() {
    for (cudaGraphExec_t g : step_graph)
      if (g) cudaGraphExecDestroy(g);
    if (hnorm) cudaFreeHost(hnorm);
    for (cudaEvent_t e : sweep_ev)
      if (e) cudaEventDestroy(e);
  }
};


// Cached per (rhs fab, phi fab, bc, options); builds coarse levels, tables and plans.
std::shared_ptr<Hierarchy> get_hierarchy(Ctx& c, FabObj& rhs, FabObj& phi, const mg_bc* bc, const SolveParams& p);
// The tables that only a solve on its own launches from (whole sweeps, residual + restriction and coarse
// cycle of one hierarchy), once per hierarchy, before its cycles are enqueued or captured: members of
// batches go without (64^3 FP64 members 3.59 -> 3.52 MB each; first batch of sixteen 32^3 mixed problems 4.0 ->
// 3.4 ms).
void prepare_alone(Ctx& c, Hierarchy& H);

// One V-cycle for the hierarchy's problem from a zero guess: phi (the caller's level-0 fab,
// ghosts included) is zeroed, then the cycle is enqueued on s; no norm is taken.
void enqueue_correction_cycle(Ctx& c, Hierarchy& H, cudaStream_t s);

}  // namespace gbmg
