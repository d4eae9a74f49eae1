// Launch of a persistent kernel that may start while the kernel ahead of it in the stream still runs (it waits for that one
// with wait_for_previous_kernel before it touches global memory), in clusters of `cluster` CTAs.
#pragma once

#include <cuda_runtime.h>

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

}  // namespace im2win
