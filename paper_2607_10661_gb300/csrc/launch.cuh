// Kernel launches chained by programmatic dependent launch (internal, not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace ptd {

// Launch with programmatic stream serialization: the grid may be placed while the stream's previous
// one drains.  The kernel calls grid_dependency_wait() before its first access to global memory,
// in every thread that makes one (so its completion implies the previous grid's), and lets its own
// successor be placed with grid_launch_dependents().  Between two kernels of a few microseconds this
// takes the launch latency (about 1.5-2 us) off the chain.
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                           unsigned cluster_x, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
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
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace ptd
