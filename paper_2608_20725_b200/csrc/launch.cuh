// Launch of a persistent kernel that may start while the kernel ahead of it in the stream still runs (it waits for that one
// with wait_for_previous_kernel before it touches global memory), in clusters of `cluster` CTAs.
#pragma once

#include <cuda_runtime.h>
#include <stdlib.h>

#include <atomic>

#include "common.cuh"

namespace im2win {

template <typename Params>
cudaError_t launch_after_previous(void (*kernel)(Params), int grid, int cluster, int threads, int smem, cudaStream_t stream,
                                  const Params& q) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, q);
}

// The same for any arguments and no cluster: the kernel may start while the one ahead of it in the stream runs its last blocks, and waits
// for it first of all that touches global memory.
// (Filter packs behind the transform, which lets them start with its last blocks: 3x3 on 64 channels at 56x56, batch 128, fp16 140.4 ->
// 139.2 us a pass, 5x5 stride 2 on 37 channels at 45x61, batch 13, fp32 41 -> 39; layers of 15 to 100 us 1.01 to 1.06 times as fast.)
template <typename... Params, typename... Args>
cudaError_t launch_early(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// Whether a cluster of z CTAs of a kernel fits the device, as far as it has been asked: 0 not yet, 1 it does, -1 it does not.
struct KnownClusters {
  std::atomic<signed char> fits[64][kMaxCtas + 1];
};

// CTAs of the clusters that share a tile: the `want` of the plan, which is made for a whole B200, or as many as the device that is there can hold,
// or 1: no clusters.  (A process may have a part of a GPU, a MIG slice or an MPS share, where the wide ones do not fit and their
// launch fails.)  Asked once for each device, kernel and size; `smem`: the most that a launch of the kernel takes.
template <typename... Params>
int ctas_that_fit(void (*kernel)(Params...), int want, int threads, int smem, KnownClusters& known) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
  int limit = kMaxCtas;
  if (const char* v = debug_getenv("IM2WIN_CLUSTER_LIMIT")) limit = atoi(v);       // testing aid: a device with room for no wider clusters
  return widest_cluster(want, [&](int z) {
    if (z > limit) return false;
    const int asked = known.fits[dev][z].load(std::memory_order_relaxed);
    if (asked != 0) return asked > 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)z; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)z, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
    known.fits[dev][z].store(clusters > 0 ? 1 : -1, std::memory_order_relaxed);
    return clusters > 0;
  });
}

}  // namespace im2win
