// lbfs_kernels.h -- launch entry points of the device kernels (host-side declarations).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lbfs_internal.cuh"

namespace lbfs {

// stage kernel (lbfs_stage.cu); prec 0 = FP64, 1 = mixed.  A strip is kStripW columns by
// `rows` rows of one case, advanced by one warp (a block of its own).
constexpr int kStripW = 26;
int stage_tile_shapes();
// rows of a strip for shape id `tile` (0: chosen from the strip-rows of all cases together)
int stage_rows(int prec, int tile, long long row_warps, int sm_count);
constexpr int kStageMinRows = 1, kStageGroup = 64;   // lowest strips; strips summed together at the step end
// half: every case streams half a cell (dts = 1/2), which selects the reconstruction
// without normal slopes at the upwind points.  one: the context's only case (host copy), or
// NULL for a batch, whose strips come from `tiles` and whose cases from `cases`.
template <class R>
cudaError_t launch_stage(int half, const StageCase<R>* one, const StageCase<R>* cases, const TileRef* tiles, int ntiles,
                         int rows, int stage, cudaStream_t st);

// potential multigrid (lbfs_potential.cu).  The extrapolation takes 32 x 32 tiles.
constexpr int kMgTX = 32, kMgTY = 32;
// The residual takes strips of kResidStripW columns by `rows` rows, one warp each, and checks
// each case once its strips are done.  first: the step's first residual (every case; later ones
// skip converged cases).  tol: the convergence test.  A case still above tol gets another cycle
// (one more vote in not_done, if given) unless it has had kmax, when it is marked as failed.
// sync: the grid barrier of launch_mg_cycles: two counters, cleared by a first check, and a mark
// that a wait of more than wait_polls polls ran out, cleared by the host.
constexpr int kResidStripW = 30, kResidMinRows = 2;
struct PotCheck {
    int first;
    double tol;
    int kmax;
    int* not_done;
    unsigned* sync;
    int wait_polls;
};
cudaError_t launch_mg_residual(int prec, const DevCase* cases, const TileRef* tiles, int n, int rows, const PotCheck& ck,
                               cudaStream_t st);
// `iters` explicit pseudo-time steps of the paper's magnetic LBFS (Eqs. 12-18) on one
// case, FP64 arithmetic; tmp holds nx*ny doubles.  2 launches per step.
cudaError_t launch_pseudo_time(int prec, const DevCase* dcase, int nx, int ny, int iters, double dtau,
                               double* tmp, cudaStream_t st);
// The V-cycle's levels from DevCase::tail down, one block per case.  A case takes it when its
// coarsest level holds at most kTailCoarsest cells, from the first level of at most kTailCells.
constexpr int kTailCells = 2048, kTailCoarsest = 1024, kPassCells = 256;
constexpr int kCoarsestMax = 4096;    // largest coarsest level accepted
// once on a context's device, before the launches below: their kernels' shared-memory limits
cudaError_t prepare_potential(int prec);
cudaError_t launch_mg_tail(int prec, const DevCase* cases, const int* case_ids, int ncases, int max_cells, int max_small,
                           cudaStream_t st);
// the coarsest level of the other cases
cudaError_t launch_mg_coarsest(const DevCase* cases, const int* case_ids, int ncases, int max_cells, cudaStream_t st);
// FP64 only: the warm start of the potential, extrapolated in time (linearly, later through three points)
cudaError_t launch_mg_extrapolate(const DevCase* cases, const TileRef* tiles, int n, cudaStream_t st);
// fused V-cycle legs over 32 x 16 tiles of one level (kFusedTX x kFusedTY), or over
// 16 x 8 tiles (small != 0) on a level whose 32 x 16 tiles would not fill the GPU
constexpr int kFusedTX = 32, kFusedTY = 16;
constexpr int kFusedSmallTX = 16, kFusedSmallTY = 8;
cudaError_t launch_mg_vdown(int prec, const DevCase* cases, const TileRef* tiles, int n, int level, int small,
                            cudaStream_t st);
cudaError_t launch_mg_vup(int prec, const DevCase* cases, const TileRef* tiles, int n, int level, int small,
                          cudaStream_t st);
constexpr int kWaitPolls = 1 << 22;   // default limit of a grid barrier's wait: seconds
// Cycles (V-cycle, residual, check) until no case needs another, in one cooperative launch of
// `blocks` blocks (at most one an SM), after a first launch_mg_residual with the same check
// and first set to 0.  max_coarsest: as for launch_mg_coarsest, 0 without such a case.
struct CycleArgs {
    const DevCase* cases;
    const TileRef* tiles[kMaxLevels];   // of the fused legs, per level with a kernel per leg
    int n_tiles[kMaxLevels], small[kMaxLevels];
    int depth;
    const int *tail, *coarsest;         // cases by how their coarse levels are solved
    int n_tail, n_coarsest, tail_cells, tail_small;
    const TileRef* strips;              // of the residual
    int n_strips, rows;
};
cudaError_t launch_mg_cycles(int prec, const CycleArgs& a, int blocks, int max_coarsest, const PotCheck& ck,
                             cudaStream_t st);

// per-case utility kernels (lbfs_fields.cu)
struct InitArgs {
    int kind;
    double radius, cx, cy, T_init, xi;
};
cudaError_t launch_init(int prec, const DevCase* dcase, int nx, int ny, InitArgs a, cudaStream_t st);
cudaError_t launch_mu_from_state(int prec, const DevCase* dcase, int nx, int ny, cudaStream_t st);
cudaError_t launch_derive_fields(int prec, const DevCase* dcase, int nx, int ny, uint32_t mask,
                                 double* out, cudaStream_t st);
cudaError_t launch_store_fields(int prec, const DevCase* dcase, int nx, int ny, uint32_t mask,
                                const double* in, cudaStream_t st);
cudaError_t launch_stats_init(int prec, const DevCase* dcase, int nx, int ny, cudaStream_t st);
// Sec. 5 diagnostics of one case: per-column scratch cols (3 nx doubles) and out5 =
// {H_m, U_max, Pe, Fo, Q_wall}; two launches.
cudaError_t launch_diagnostics(int prec, const DevCase* dcase, int nx, double R0, double* cols,
                               double* out5, cudaStream_t st);

}  // namespace lbfs
