// Launches that may begin while the kernel before them in the stream is still running.
#pragma once

#include <cuda_runtime.h>

namespace sigattn {

// Programmatic stream serialisation: once every thread block of the preceding kernel has called
// grid_dependency_trigger() (or ended), this kernel's blocks may be scheduled; each of them runs its set-up and then
// waits in grid_dependency_wait() until the preceding kernel has completed and its writes are visible.  Every kernel
// launched this way calls both, with all threads, before it touches global memory, so that completion stays
// transitive along the stream.  Preceding work of any other kind (copies, clears, kernels of other libraries) is
// waited for as usual.  A kernel that uses tensor memory triggers only after its own allocation has succeeded (behind a
// __syncthreads): a block of the next kernel, which holds what it allocates until this kernel ends, must not be able
// to take it first.  What it saves is the launch latency and the set-up (barriers, tensor memory) of kernels that
// follow one another, 1 to 2.5 us of each short call.
template <typename... KernelArgs, typename... Args>
cudaError_t launch_after(void (*kernel)(KernelArgs...), dim3 grid, unsigned threads, size_t smem_bytes,
                         cudaStream_t stream, unsigned cluster_x, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster_x;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster_x > 0 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

#ifdef __CUDACC__
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

}  // namespace sigattn
