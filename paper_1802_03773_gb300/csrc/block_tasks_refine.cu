// Instantiation of the warp-task refinement kernel with the compensated-float residual (one
// kernel per translation unit, so that the variants compile in parallel).
#include "block_tasks.cuh"

namespace qrkit {
namespace tasks {

template <int RES>
cudaError_t refine_setup(size_t smem, int threads, int* per_sm) {
  auto k = block_task_refine_kernel<RES, false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k, threads, smem);
}

template <int RES>
cudaError_t refine_launch(const RefineTaskArgs& A, unsigned grid, int threads, size_t smem, cudaStream_t st,
                          bool chained) {
  if (chained) return chain_launch(st, grid, threads, smem, block_task_refine_kernel<RES, true>, A);
  block_task_refine_kernel<RES, false><<<grid, threads, smem, st>>>(A);
  return cudaGetLastError();
}

template cudaError_t refine_setup<0>(size_t, int, int*);
template cudaError_t refine_launch<0>(const RefineTaskArgs&, unsigned, int, size_t, cudaStream_t, bool);

}  // namespace tasks
}  // namespace qrkit
