// Launches that begin while the kernel before them ends (programmatic dependent launch).
//
// A kernel whose first statement is chain_wait() may be launched by chain_launch: its blocks are set up as those of
// the kernel before it end, and wait there until that kernel has ended altogether and its writes are
// visible.  What follows the wait runs as after an ordinary launch, so the order of a stream's work is the
// same; what overlaps is the launch.  Measured, all launches of a call chained: one
// million columns of a banded system (68 launches) 975 -> 827 us, 100,000 blocks with 5 shared columns 196 -> 157 us,
// 100,000 blocks with 128 shared columns 1658 -> 1540 us.
//
// The wait is for the one kernel before, so the order holds only if that kernel waited for its own predecessor.  This
// library's kernels do; a caller's need not (a kernel launched this way that never waits may end before the one that
// writes our input).  The first launch of every call is therefore an ordinary one (start_launch, or a
// memset or copy before it), which the stream orders behind everything.
//
// One kernel waits at its end instead: block_task_kernel<.., 2, true>, which runs beside the kernel launched before it
// in the same call, has its own tasks and outputs, and reads nothing that kernel writes.
//
// Allowing the next launch earlier, from the kernel's first statement (chain_next), only pays for kernels that
// leave most of the chip idle: blocks that wait take slots and keep the scheduler busy.
#pragma once

#include <cuda_runtime.h>

namespace qrkit {
namespace dev {

// The next kernel may be set up (once every block has called this or ended).
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;"); }
// The kernel before this one has ended (nothing to wait for after an ordinary launch).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace dev

template <typename... P, typename... A>
cudaError_t launch_kernel(bool chained, cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*kernel)(P...),
                          A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = chained ? &attr : nullptr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Launch of a kernel that begins with chain_wait(), after another of the same call.
template <typename... P, typename... A>
cudaError_t chain_launch(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*kernel)(P...), A... args) {
  return launch_kernel(true, st, grid, block, smem, kernel, args...);
}
// The first launch of a call.
template <typename... P, typename... A>
cudaError_t start_launch(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*kernel)(P...), A... args) {
  return launch_kernel(false, st, grid, block, smem, kernel, args...);
}

}  // namespace qrkit
