// Launches of the kernels that follow one another in a run (programmatic
// dependent launch): a step's blocks may take their places, and its launch
// latency may pass, while the step before drains.  Every kernel launched so
// begins with chain_begin(p), which waits until the work before it in the
// stream has finished and its writes are visible; the kernel reads through the
// pointer that it returns, so that no load can be moved ahead of the wait.  As
// each waits for its predecessor to finish, the order along the stream is that
// of plain launches.
//
// Chained: the steps of one simulation in one and two dimensions (512 x 512
// bilinear FP32: 14.4 -> 13.0 us per step; adjoint run of 96 steps at 512 x 512:
// 4.91 -> 4.49 ms; a grid of many waves gains 1-2 %).  Plain (Scalars::plain):
// the (3+1)-d steps, whose tens of waves lose 1 % to the next grid's blocks
// resuming in step, and the batch's concurrent chains (3 %: waiting blocks hold
// places that another chain could use).
#pragma once
#include <cuda_runtime.h>

namespace rlbm {

#ifdef __CUDACC__
template <typename T>
__device__ __forceinline__ T* chain_begin(T* p) {
  asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" : "+l"(p) : : "memory");
  return p;
}

// another pointer that is read after chain_begin()
template <typename T>
__device__ __forceinline__ T* chained(T* p) {
  asm volatile("" : "+l"(p) : : "memory");
  return p;
}

template <typename... P, typename... A>
cudaError_t launch_chained_clusters(bool chained, int cluster, void (*kernel)(P...), dim3 grid, dim3 block, size_t shared,
                                    cudaStream_t st, const A&... args) {
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (chained) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cluster;
    attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = shared;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename... P, typename... A>
cudaError_t launch_chained(bool chained, void (*kernel)(P...), dim3 grid, dim3 block, size_t shared, cudaStream_t st,
                           const A&... args) {
  return launch_chained_clusters(chained, 1, kernel, grid, block, shared, st, args...);
}
#endif

}  // namespace rlbm
