// Launches with programmatic dependent launch: a kernel of a pass may be set up (its CTAs placed, barriers
// initialised, tensor memory taken) while the kernel before it drains, and waits for that kernel's results at
// pdl_wait().  Every kernel launched this way calls pdl_wait() in every thread that touches global memory, before it
// does, so completion stays transitive along the stream; pdl_trigger() lets the next kernel start its own set-up.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <utility>

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t smat_launch_pdl(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
