// Kernel launches.
#pragma once
#include <cuda_runtime.h>

namespace tq {

// A launch that may start while the previous kernel of the stream still runs
// (programmatic dependent launch): the kernel waits for it (grid_dep_wait,
// tq_sm100.cuh) before it reads anything.  With cluster > 1 the grid is made
// of clusters of that many CTAs.
template <class... P, class... A>
inline cudaError_t launch_dependent_cluster(void (*kern)(P...), dim3 grid, int cluster, int threads, int smem,
                                            cudaStream_t s, const A &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<const P &>(args)...);
}
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, int threads, cudaStream_t s, const A &...args) {
  return launch_dependent_cluster(kern, grid, 1, threads, 0, s, args...);
}
// The same with a kernel's most shared memory (always the same for a kernel:
// several threads may set it at once).
template <class... P, class... A>
inline cudaError_t launch_big_smem(void (*kern)(P...), int ctas, int threads, int smem, cudaStream_t s,
                                   const A &...args) {
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_dependent_cluster(kern, dim3(ctas), 1, threads, smem, s, args...);
}

}  // namespace tq
