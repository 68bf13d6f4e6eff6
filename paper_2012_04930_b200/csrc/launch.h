// Kernel launches whose start overlaps the end of the kernel before them on the stream (programmatic dependent launch):
// the training steps are chains of kernels of a few microseconds, and bringing the next one up costs as much as many of
// them run.  Every kernel launched this way waits for its predecessors before it touches global memory
// (wait_for_predecessors, first thing or after a prologue on shared and tensor memory) and then lets its own successor
// come up.
#pragma once
#include <cuda_runtime.h>

namespace gcnsa {

#ifdef __CUDACC__
__device__ __forceinline__ void wait_for_predecessors() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Up to this many blocks.  A kernel of hundreds of microseconds gains nothing, and one that lives on the order in which its
// blocks are handed out loses: spmm_rows over 269 498 rows (F' = 256, 30 000 blocks) took 572 us launched plainly, 695
// this way.
constexpr long long kOverlapBlocks = 8 * 148;

template <class... P, class... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t shared, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = shared;
  c.stream = stream;
  cudaLaunchAttribute a;
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = (long long)grid.x * grid.y * grid.z <= kOverlapBlocks ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// the same in clusters of `cluster` consecutive blocks
template <class... P, class... A>
inline cudaError_t launch_cluster(int cluster, void (*kernel)(P...), dim3 grid, dim3 block, size_t shared, cudaStream_t stream,
                                  A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = shared;
  c.stream = stream;
  cudaLaunchAttribute a[2];
  a[0].id = cudaLaunchAttributeClusterDimension;
  a[0].val.clusterDim.x = cluster;
  a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
  a[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a[1].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = a;
  c.numAttrs = (long long)grid.x * grid.y * grid.z <= kOverlapBlocks ? 2 : 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
#endif

}  // namespace gcnsa
