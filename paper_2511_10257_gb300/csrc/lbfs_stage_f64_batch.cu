// lbfs_stage_f64_batch.cu -- the stage kernel in FP64, a batch of cases.
#define LBFS_STAGE_DEFINE 1
#include "lbfs_stage.cuh"

namespace lbfs {

template cudaError_t stage_launch<double, true, false>(const StageCase<double>&, const StageCase<double>*, const TileRef*, int, int, int,
                                                cudaStream_t);
template cudaError_t stage_launch<double, false, false>(const StageCase<double>&, const StageCase<double>*, const TileRef*, int, int, int,
                                                 cudaStream_t);

}  // namespace lbfs
