// lbfs_stage_f32_batch.cu -- the stage kernel in mixed precision, a batch of cases.
#define LBFS_STAGE_DEFINE 1
#include "lbfs_stage.cuh"

namespace lbfs {

template cudaError_t stage_launch<float, true, false>(const StageCase<float>&, const StageCase<float>*, const TileRef*, int, int, int,
                                                cudaStream_t);
template cudaError_t stage_launch<float, false, false>(const StageCase<float>&, const StageCase<float>*, const TileRef*, int, int, int,
                                                 cudaStream_t);

}  // namespace lbfs
