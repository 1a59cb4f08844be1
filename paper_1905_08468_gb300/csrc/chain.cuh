// Launches of an iteration's kernels back to back (programmatic dependent
// launch): the next kernel is made ready while the one before it runs, and its
// CTAs are placed as soon as that one's have left; chain_enter(), the first
// thing a kernel of the chain does with memory that another one writes, waits
// until the kernel before has finished and its results are visible.  This takes
// part of the launch latency out of every boundary: 64 x 64 x 8 (10 kernels an
// iteration, 8 since the gradient is one) 43.5 -> 39 us an iteration, 256 x 256 x 37 1-2 percent, large cubes
// unchanged.  No kernel triggers its dependents early: waiting CTAs then hold
// registers and shared memory beside the running kernel's last waves (1024 x
// 1024 x 256: 196 -> 210 ms a pass, triggered before or after the wait).
// A kernel launched otherwise waits for nothing more than the stream's order.
#pragma once

#include <cuda_runtime.h>

namespace muffin {

__device__ __forceinline__ void chain_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
cudaError_t launch_chain(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                         cudaStream_t st, A... args) {
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

}  // namespace muffin
