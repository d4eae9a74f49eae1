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

// A filter pack, launched early and spread over the SMs (spread_smem): its blocks are small and none has much to do.
// (Passes that pack, without / with: 7x7 on 181 -> 32 channels at 10x10, batch 64, channel-innermost, 45.1 -> 39.1 us, 5x5 on 512 -> 22
// at 12x12 56.2 -> 49.2; 362 drawn channel-innermost ones 1.014 on average, 413 others 1.003.  The other way round where the output bounds the
// pass and CTAs that start in another order write it worse: 3x3 on 3 -> 236 channels at 118x118, batch 106, 443 -> 467.)
template <auto kernel, typename... Args>
cudaError_t launch_pack(dim3 grid, int threads, size_t smem, cudaStream_t stream, const Args&... args) {
  static bool attr_done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr_done[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSpread);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  return launch_early(kernel, grid, threads, spread_smem((int64_t)grid.x * grid.y, threads, smem), stream, args...);
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
