// Bulk delete (Sec. 4.1 upkeep; Sec. 4.2: a dead entry of the key is removed as
// well, and reported as not found).
//
// Kernels, in stream order, after the workspace clear:
//   delete_kernel  per key: its owner (dedup.cuh), found in the table by the
//                  lookup's line fetches (probe.cuh), removes the entry;
//   delete_settle  the followers before their owner in the batch: the lowest
//                  index of each group takes over its outcome.
#include "chain_launch.h"
#include "dedup.cuh"
#include "probe.cuh"

namespace ckpp {

namespace {

constexpr int kDeleteThreads = 64;  // 1M absent keys: 55.9 us, with 128 56.9, with 32 58.6
constexpr int kDeleteClusterThreads = 256;
constexpr int kSettleThreads = 256;

// One warp, 32 keys (every thread of the block calls this). The set's CAS is requested before the bucket lines and
// looked at after them. The primary's and secondary's lines come whole (one
// request each, with the entries of the first slots), as in a lookup: reading
// a bucket's header and then the key of a matching slot were two random
// accesses per key. It is bound by line requests: 1.6 per key read, one for the
// ctrl word's AND, and two more atomics for each displaced entry. Whole calls
// against a dedup kernel and lane-by-lane reads: 1M keys of 134M slots 125 ->
// 116 us, of 34M slots with timers 134 -> 103 us, 256K keys 46 -> 38 us.
template <int kTM>
__device__ __forceinline__ void delete_chunk(const TableSet& ts, const uint8_t* __restrict__ keys, uint64_t i64,
                                             uint64_t n, uint32_t now, uint8_t* __restrict__ status,
                                             const Workspace& ws, WarpStage<1>& stage, BlockLists<1>& lists) {
  const uint32_t i = (uint32_t)i64;
  bool act[1] = {i64 < n};
  if (act[0] && !ts.valid(i)) {
    status[i] = kStNoTable;
    act[0] = false;
  }
  TableView t{};
  Key k{0, 0};
  uint32_t tid = 0;
  if (act[0]) {
    t = ts.of(i);
    tid = ts.id(i);
    k = load_key(keys, i);
  }
  Probe p[1];
  uint64_t h1;
  probe_init(p[0], k, t.buckets, t.nb, t.seed, t.timers, h1);
  SetProbe sp{0, 0, kEmpty};
  if (act[0]) sp = set_probe(ws, h1, tid, i);
  run_probes<kBloom, false, 1, kTM>(p, act, now, stage);
  bool follows = false;
  uint32_t owner = kNoIndex;
  if (act[0]) {
    owner = set_owner(ws, ts, keys, k, tid, i, sp);
    follows = owner != i;
    if (!follows) {
      if (p[0].hs != kNoSlot) {  // stored, alive (found) or dead
        const uint32_t slot = p[0].hs;
        atomicAnd(ctrl_ptr(t, p[0].hb), ~((1u << slot) | (1u << (kInsecShift + slot))));
        // Sec. 4.1: removing a displaced key decrements its primary's counter; at
        // zero the filter is reset. No filter bit is set during a delete batch.
        if (p[0].hb == p[0].b2 && atomicSub(moved_ptr(t, p[0].b1), 1u) == 1u)
          atomicExch(reinterpret_cast<unsigned long long*>(bloom_ptr(t, p[0].b1)), 0ull);
      }
      status[i] = p[0].found ? kStDeleted : kStNotFound;
    }
  }
  // a repeated key is not found, unless it turns out to be its group's lowest index
  if (follows) status[i] = kStNotFound;
  const bool before = follows && i < owner;
  uint32_t at[1];
  lists_append<1>(lists, {ws.counters + kCntFollowers}, {before}, at);
  if (before) write_follower(ws, at[0], i, owner);
}

template <int kTM>
__global__ void __launch_bounds__(kDeleteThreads) delete_kernel(TableSet ts, const uint8_t* __restrict__ keys,
                                                                uint64_t n, uint32_t now,
                                                                uint8_t* __restrict__ status, Workspace ws) {
  __shared__ WarpStage<1> stage[kDeleteThreads / 32];
  __shared__ BlockLists<1> lists;
  lists_init(lists);
  pdl_wait();
  delete_chunk<kTM>(ts, keys, blockIdx.x * (uint64_t)kDeleteThreads + threadIdx.x, n, now, status, ws,
                    stage[threadIdx.x >> 5], lists);
}

// A group's lowest index takes over DELETED from its owner.
__device__ __forceinline__ void settle_range(uint8_t* __restrict__ status, const Workspace& ws, uint32_t followers,
                                             uint32_t worker, uint32_t workers) {
  for (uint32_t j = worker; j < followers; j += workers) {
    const uint2 f = ws.followers[j];
    if (f.x == ws.range[f.y].x && status[f.y] == kStDeleted) {
      status[f.x] = kStDeleted;
      status[f.y] = kStNotFound;
    }
  }
}

__global__ void __launch_bounds__(kSettleThreads) delete_settle(uint8_t* __restrict__ status, Workspace ws) {
  pdl_wait();
  settle_range(status, ws, ld32_cg(ws.counters + kCntFollowers), blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// A small batch in one launch of one cluster (as insert_cluster).
template <int kTM>
__global__ void __launch_bounds__(kDeleteClusterThreads) delete_cluster(TableSet ts, const uint8_t* __restrict__ keys,
                                                                 uint64_t n, uint32_t now,
                                                                 uint8_t* __restrict__ status, Workspace caller_ws) {
  __shared__ WarpStage<1> stage[kDeleteClusterThreads / 32];
  __shared__ BlockLists<1> lists;
  __shared__ OneBlockSet one_set;
  __shared__ OneBlockGroups one_groups;
  const uint32_t tid = blockIdx.x * kDeleteClusterThreads + threadIdx.x, threads = gridDim.x * kDeleteClusterThreads;
  const Workspace ws = gridDim.x == 1 ? in_shared(caller_ws, one_set, one_groups) : caller_ws;
  lists_init(lists);
  pdl_wait();
  clear_workspace(ws, tid, threads);
  cluster_barrier();
  for (uint32_t first = blockIdx.x * kDeleteClusterThreads; first < n; first += threads)
    delete_chunk<kTM>(ts, keys, first + threadIdx.x, n, now, status, ws, stage[threadIdx.x >> 5], lists);
  cluster_barrier();
  settle_range(status, ws, ld32_cg(ws.counters + kCntFollowers), tid, threads);
}
static_assert(kOneBlockKeys == kDeleteClusterThreads, "cluster_blocks gives batches that fit one block a cluster of one");

}  // namespace

cudaError_t launch_delete(const TableSet& ts, const uint8_t* keys, uint64_t n, uint32_t now, uint8_t* status,
                          const Workspace& ws, cudaStream_t s) {
  if (n <= kClusterKeys) {
    auto kernel = !ts.any_timers ? delete_cluster<kNoTimers> : ts.views ? delete_cluster<kTimersPerKey>
                                                                       : delete_cluster<kWithTimers>;
    return launch_cluster(kernel, cluster_blocks(n, kDeleteClusterThreads), kDeleteClusterThreads, 0, s, ts, keys, n, now, status,
                          ws);
  }
  const unsigned grid = grid_for(n, kDeleteThreads);
  cudaError_t e = launch_workspace_clear(ws, s);
  if (e != cudaSuccess) return e;
  if (!ts.any_timers) {
    e = launch_chained(delete_kernel<kNoTimers>, grid, kDeleteThreads, s, ts, keys, n, now, status, ws);
  } else if (!ts.views) {
    e = launch_chained(delete_kernel<kWithTimers>, grid, kDeleteThreads, s, ts, keys, n, now, status, ws);
  } else {
    e = launch_chained(delete_kernel<kTimersPerKey>, grid, kDeleteThreads, s, ts, keys, n, now, status, ws);
  }
  if (e != cudaSuccess) return e;
  const unsigned most = 2u * (unsigned)device_sm_count(), want = grid_for(n, kSettleThreads);
  return launch_chained(delete_settle, want < most ? want : most, kSettleThreads, s, status, ws);
}

}  // namespace ckpp
