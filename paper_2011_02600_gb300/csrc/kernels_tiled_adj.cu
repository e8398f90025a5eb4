// The tiled stage kernel (kernels_tiled.cuh): the FP32 adjoint passes.
#include "kernels_tiled.cuh"

namespace sbp {

template <>
cudaError_t launch_adjoint_tiled<float>(const StageArgs<float>& A, int order, int pass, const TmaSet& tm, cudaStream_t st) {
  if (pass == 1) {
    if (!A.ubar_out || (A.mode != kModeRhs && !A.wbar)) return cudaErrorInvalidValue;
    return launch_kind<float, 1>(A, order, tm, st);
  }
  if (pass == 2) {
    if (!A.wbar || !A.yhat || !A.rlmj || !A.grad) return cudaErrorInvalidValue;
    return launch_kind<float, 2>(A, order, tm, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace sbp
