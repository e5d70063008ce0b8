// Launches with programmatic dependent launch: a kernel of a pass may be set up (its CTAs placed, barriers
// initialised, tensor memory taken) while the kernel before it drains, and waits for that kernel's results at
// pdl_wait().  Every kernel launched this way calls pdl_wait() in every thread that touches global memory, before it
// does, and in at least one thread of every CTA, also of one that has nothing to do: a launch whose CTAs all leave without
// it completes beside the kernel before, and completion would no longer be transitive along the stream.  pdl_trigger()
// lets the next kernel start its own set-up.  Three rules follow.
// A bounded wait (mbar_wait) for anything that another thread brings about after its pdl_wait() comes after a pdl_wait()
// of its own: the limit counts this kernel's time, not what is left of the kernel before.
// A kernel that takes tensor memory triggers only after it has it: the next kernel's CTAs start once all of this one's have
// triggered, and a CTA that took the columns first and then waited for this kernel would never give them back.
// Data of earlier kernels is read with plain loads, not through __ldg or const __restrict__ pointers: the compiler may
// move such loads of "constant" memory above the wait.
#pragma once
#include <cuda_runtime.h>

#include <utility>

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// cluster_x > 1: thread-block clusters of that many neighbouring CTAs along x.
template <typename... KArgs, typename... Args>
cudaError_t smat_launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, unsigned cluster_x,
                                    cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster_x;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster_x > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t smat_launch_pdl(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, Args&&... args) {
  return smat_launch_pdl_cluster(kernel, grid, block, smem, 1u, st, std::forward<Args>(args)...);
}
