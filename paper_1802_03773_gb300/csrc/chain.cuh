// Launches that begin while the kernel before them ends (programmatic dependent launch).
//
// A kernel whose first statement is chain_wait() may be launched by chain_launch: its blocks are set up as those of
// the kernel before it end, and wait there until that kernel has ended altogether and its writes are
// visible.  What follows the wait runs as after an ordinary launch, so the order of a stream's work is the
// same; what overlaps is the launch.  Allowing the next launch earlier, from the kernel's first statement
// (chain_next), only pays for kernels that leave most of the chip idle: blocks that wait take slots and keep the
// scheduler busy.  Measured, all launches of a call chained: one
// million columns of a banded system (68 launches) 975 -> 827 us, 100,000 blocks with 5 shared columns 196 -> 157 us,
// 100,000 blocks with 128 shared columns 1658 -> 1540 us.
#pragma once

#include <cuda_runtime.h>

namespace qrkit {
namespace dev {

// The next kernel may be set up (once every block has called this or ended).
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;"); }
// The kernel before this one has ended (nothing to wait for after an ordinary launch).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace dev

// Launch of a kernel that begins with chain_begin() (an ordinary launch needs no such kernel).
template <typename... P, typename... A>
cudaError_t chain_launch(cudaStream_t st, dim3 grid, dim3 block, size_t smem, void (*kernel)(P...), A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace qrkit
