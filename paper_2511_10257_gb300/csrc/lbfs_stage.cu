// lbfs_stage.cu -- launches of the stage kernel.
#include "lbfs_kernels.h"
#include "lbfs_stage.cuh"

namespace lbfs {

// Strip heights by id; id 0 leaves the choice to stage_rows' rule.
static constexpr int kShapes = 13;
static constexpr int kShapeRows[kShapes] = {0, 128, 96, 64, 48, 32, 24, 16, 12, 8, 4, 2, 1};

int stage_tile_shapes() { return kShapes; }

// A strip costs its rows plus about 2.4 more (the rows at its ends that serve only its
// neighbours), so tall strips are cheaper per cell, and as long as all strips run at once the
// lowest ones finish first.  Hence the lowest strips that still fit the GPU in one wave (12
// warps an SM in mixed precision; in FP64 4, one per FP64 pipe), up to 24 rows (32 in FP64),
// from where the ends no longer matter.  Measured, us per stage-2 launch in mixed precision:
// 128x64: 1 row 10.8, 2 rows 12.4, 4 rows 14.5; 512x256: 2 rows 19.0, 4 rows 17.3, 8 rows 22.7;
// 1024x512: 8 rows 35.4, 12 rows 33.3, 16 rows 41.7; 4096x2048: 16 rows 280, 24 rows 277,
// 32 rows 278, 64 rows 308.  FP64: 128x64: 1 row 60, 2 rows 79; 512x256: 8 rows 287, 12 rows
// 281, 16 rows 360; 4096x2048 (ms): 16 rows 11.7, 32 rows 11.3, 64 rows 11.7.
int stage_rows(int prec, int tile, long long row_warps, int sm_count) {
    if (tile > 0 && tile < kShapes) return kShapeRows[tile];
    const long long wave = (long long)sm_count * (prec == 0 ? 4 : 12);
    const int most = prec == 0 ? 32 : 24;
    for (int i = kShapes - 1; i > 0; --i)
        if (kShapeRows[i] >= most || row_warps <= wave * kShapeRows[i]) return kShapeRows[i];
    return most;
}

template <class R>
cudaError_t launch_stage(int half, const StageCase<R>* one, const StageCase<R>* cases, const TileRef* tiles, int ntiles,
                         int rows, int stage, cudaStream_t st) {
    if (ntiles <= 0) return cudaSuccess;
    if (one) return half ? stage_launch<R, true, true>(*one, cases, tiles, ntiles, rows, stage, st)
                         : stage_launch<R, false, true>(*one, cases, tiles, ntiles, rows, stage, st);
    const StageCase<R> none{};
    return half ? stage_launch<R, true, false>(none, cases, tiles, ntiles, rows, stage, st)
                : stage_launch<R, false, false>(none, cases, tiles, ntiles, rows, stage, st);
}
template cudaError_t launch_stage<float>(int, const StageCase<float>*, const StageCase<float>*, const TileRef*, int, int, int,
                                         cudaStream_t);
template cudaError_t launch_stage<double>(int, const StageCase<double>*, const StageCase<double>*, const TileRef*, int, int,
                                          int, cudaStream_t);

}  // namespace lbfs
