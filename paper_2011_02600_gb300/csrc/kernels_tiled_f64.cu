// The tiled stage kernel (kernels_tiled.cuh): the FP64 forward stage.
#include "kernels_tiled.cuh"

namespace sbp {

template <>
cudaError_t launch_stage_tiled<double>(const StageArgs<double>& A, int order, const TmaSet& tm, cudaStream_t st) {
  return launch_kind<double, 0>(A, order, tm, st);
}

}  // namespace sbp
