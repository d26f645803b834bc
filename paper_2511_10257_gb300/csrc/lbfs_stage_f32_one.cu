// lbfs_stage_f32_one.cu -- the stage kernel in mixed precision, one case.
#define LBFS_STAGE_DEFINE 1
#include "lbfs_stage.cuh"

namespace lbfs {

template cudaError_t stage_launch<float, true, true>(const StageCase<float>&, const StageCase<float>*, const TileRef*, int, int, int,
                                                cudaStream_t);
template cudaError_t stage_launch<float, false, true>(const StageCase<float>&, const StageCase<float>*, const TileRef*, int, int, int,
                                                 cudaStream_t);

}  // namespace lbfs
