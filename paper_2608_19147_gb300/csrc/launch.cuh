// Launches that may begin while the kernel before them in the stream ends.
#pragma once
#include <utility>

#include "common.cuh"

namespace shard {

// Launches `kern` with programmatic dependent launch: its CTAs may take their
// places once every CTA of the preceding kernel has called
// pdl_launch_dependents() (or ended). The kernel calls pdl_wait() before its
// first access to anything another kernel writes or reads.
template <class... Params, class... Args>
cudaError_t launch_behind(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

}  // namespace shard
