// Host side of a call that runs as a chain of kernels on one stream (insert,
// delete): each kernel is launched with programmatic stream serialization and
// waits for its predecessor in its first instruction (pdl_wait in mutate.cuh), so
// that the GPU schedules it while the predecessor drains. That includes the
// chain's first, the workspace clear, whose predecessor is whatever the stream
// holds: 2 us less per call than a clear launched without (delete of 4K absent
// keys 10.4 -> 8.6 us). It releases its successor only after its own wait, so a
// call's other kernels start when all that was queued before the call is
// complete, and may read the batch through the read-only path.
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

// Batches this small run as one launch of one cluster, without a chain. Insert
// and delete of n keys, back to back through the C ABI, 2^17 buckets at load
// 0.8, a tenth of the keys repeated, chain / cluster in us: 1 key 20.5 / 12.5,
// 64 29.1 / 20.1, 256 29.8 / 22.7, 1024 36.1 / 28.8, 2048 43.2 / 35.1, 3072 42.4
// / 47.1: beyond 2048 keys a cluster's 2048 threads take several each.
constexpr uint64_t kClusterKeys = 2048;
constexpr unsigned kClusterMaxBlocks = 8;  // the portable cluster size

inline unsigned cluster_blocks(uint64_t n, int threads) {
  const unsigned want = grid_for(n, threads);
  unsigned blocks = 1;
  while (blocks < want && blocks < kClusterMaxBlocks) blocks *= 2;
  return blocks;
}

template <typename... Params, typename... Args>
cudaError_t launch_cluster(void (*kernel)(Params...), unsigned blocks, unsigned block, size_t smem,
                           cudaStream_t s, Args... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = blocks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace ckpp
