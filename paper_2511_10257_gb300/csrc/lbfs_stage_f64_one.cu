// lbfs_stage_f64_one.cu -- the stage kernel in FP64, one case.
#define LBFS_STAGE_DEFINE 1
#include "lbfs_stage.cuh"

namespace lbfs {

template cudaError_t stage_launch<double, true, true>(const StageCase<double>&, const StageCase<double>*, const TileRef*, int, int, int,
                                                cudaStream_t);
template cudaError_t stage_launch<double, false, true>(const StageCase<double>&, const StageCase<double>*, const TileRef*, int, int, int,
                                                 cudaStream_t);

}  // namespace lbfs
