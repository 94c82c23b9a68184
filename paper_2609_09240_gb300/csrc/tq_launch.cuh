// Kernel launches.
#pragma once
#include <atomic>

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

// Clusters of `cluster` (up to 16) CTAs of KERN, each with `smem` bytes of
// dynamic shared memory, that the current device runs at once; 0 where it
// holds none or that cannot be told (a partition whose GPCs have fewer SMs, a
// failing query: its error does not stay behind for the caller's next check).
// A kernel asks for one smem only; devices are asked once.
template <auto KERN>
int clusters_at_once(int cluster, int threads, int smem) {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices][17];  // clusters + 1, 0: not asked yet
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
  std::atomic<int> *slot = dev >= 0 && dev < kDevices ? &known[dev][cluster] : nullptr;
  if (slot && slot->load(std::memory_order_relaxed)) return slot->load(std::memory_order_relaxed) - 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cluster);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (dev < 0 || cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      (cluster > 8 && cudaFuncSetAttribute(KERN, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
      cudaOccupancyMaxActiveClusters(&n, KERN, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    n = 0;
  }
  if (slot) slot->store(n + 1, std::memory_order_relaxed);
  return n;
}

}  // namespace tq
