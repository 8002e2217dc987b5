// Host side of the batch calls' launches. Every kernel, the first of a call too
// (its predecessor is whatever the stream holds), is launched with programmatic
// stream serialization and waits for its predecessor in its first instruction
// (pdl_wait in ckpp_device.cuh): its launch is prepared while the predecessor
// runs. Per call, against a plain launch of the first kernel: a lookup of 1M keys
// in a 32 MB table 18.5 -> 16.1 us, of 50K in a 1 GB table 6.3 -> 4.5, a batched
// launch of 48 jobs 8.3 -> 6.0, insert and delete of one key 12.5 -> 8.8, delete
// of 4K absent keys 10.4 -> 8.1.
// No kernel releases its successor before its own end: blocks of a kernel that
// become resident beside another's keep that one's split of L1 and shared memory,
// and hand it on to the kernels after them (a million keys inserted, looked up
// and deleted: 375 us with early releases everywhere, 342 without any in a call's
// last kernel, 336 without any).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace ckpp {

inline unsigned grid_for(uint64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <typename... Params, typename... Args>
cudaError_t launch_chained_smem(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                                Args... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), unsigned grid, unsigned block, cudaStream_t s, Args... args) {
  return launch_chained_smem(kernel, grid, block, 0, s, args...);
}

// Batches this small run on one cluster, without a chain (inserts of more than 64
// keys with one launch after it, insert.cu, which is not in these figures). Insert
// and delete of n keys, back to back through the C ABI, 2^17 buckets at load
// 0.8, a tenth of the keys repeated, chain / cluster in us: 768 keys 30.9 /
// 24.3, 1024 31.0 / 24.1, 1536 34.9 / 28.0, 2048 35.9 / 29.0, 3072 34.4 / 38.3,
// 4096 34.9 / 39.9: beyond 2048 keys a cluster's 2048 threads take several each.
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
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = blocks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace ckpp
