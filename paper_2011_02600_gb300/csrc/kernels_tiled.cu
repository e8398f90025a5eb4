// The tiled stage kernel (kernels_tiled.cuh): the FP32 forward stage, and the self-test of its
// bounded wait.  The FP64 stage and the adjoint passes are in translation units of their own, so
// that they compile in parallel.
#include "kernels_tiled.cuh"

namespace sbp {

template <>
cudaError_t launch_stage_tiled<float>(const StageArgs<float>& A, int order, const TmaSet& tm, cudaStream_t st) {
  return launch_kind<float, 0>(A, order, tm, st);
}

// Self-test of the bounded wait used by the tiled kernel: one thread initialises an mbarrier
// that expects one arrival, nothing arrives, and the wait gives up after `polls` polls and
// records SBP_STATUS_TIMEOUT in the status word, exactly as the stage kernel does when a tile
// copy never lands.  The barrier lives in shared memory; nothing is left in flight.
__global__ void wait_selftest_kernel(unsigned polls, unsigned* status) {
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  fence_mbar_init();
  if (!mbar_wait_bounded(&bar, 0, polls)) atomicOr(status, 8u);
}

cudaError_t launch_wait_selftest(unsigned polls, unsigned* status, cudaStream_t st) {
  wait_selftest_kernel<<<1, 32, 0, st>>>(polls, status);
  return cudaGetLastError();
}

}  // namespace sbp
