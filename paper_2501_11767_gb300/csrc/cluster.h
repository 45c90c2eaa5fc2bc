// Launches of kernels that run as thread-block clusters.
#pragma once

#include "internal.h"

namespace chnss {

// Allow clusters of up to 16 blocks and `smem` bytes of dynamic shared memory
// for a kernel: once per kernel and device (the attributes are the device's).
template <auto Kernel>
void allow_cluster(size_t smem) {
  constexpr int kDevs = 64;
  static std::atomic<bool> done[kDevs];
  int dev = 0;
  CHNSS_CK(cudaGetDevice(&dev));
  if (dev >= 0 && dev < kDevs && done[dev].load(std::memory_order_acquire)) return;
  CHNSS_CK(cudaFuncSetAttribute(Kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  CHNSS_CK(cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  if (dev >= 0 && dev < kDevs) done[dev].store(true, std::memory_order_release);
}

// `clusters` clusters of `ctas` blocks each
template <typename... P, typename... A>
void launch_cluster(void (*kernel)(P...), int ctas, int clusters, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ctas * clusters));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  CHNSS_CK(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
}

// Whether the device can hold one such cluster: 16 blocks are more than the
// portable 8, and a partition of a device, or one with smaller groups of
// multiprocessors, may have no place for them.  Asked when a plan is made;
// where the answer is no, the per-launch or one-block form runs instead.
template <auto Kernel>
bool cluster_runs(int ctas, int threads, size_t smem, size_t most) {
  int clusters = 0;
  try {
    allow_cluster<Kernel>(most);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    CHNSS_CK(cudaOccupancyMaxActiveClusters(&clusters, Kernel, &cfg));
  } catch (const Error &) {
    cudaGetLastError();
    return false;
  }
  return clusters > 0;
}

}  // namespace chnss
