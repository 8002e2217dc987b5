// Host side of a call that runs as a chain of kernels on one stream (insert,
// delete): each kernel after the first is launched with programmatic stream
// serialization and waits for its predecessor in its first instruction
// (pdl_wait in mutate.cuh), so that the GPU schedules it while the predecessor
// drains.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace ckpp {

inline unsigned grid_for(uint64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), unsigned grid, unsigned block, cudaStream_t s, Args... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace ckpp
