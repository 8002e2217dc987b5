// Bulk delete (Sec. 4.1 upkeep; Sec. 4.2: a dead entry of the key is removed as
// well, and reported as not found).
//
// Kernels, in stream order, after the workspace clear:
//   delete_kernel  per key: its owner (dedup.cuh), found in the table by the
//                  lookup's line fetches (probe.cuh), removes the entry;
//   delete_ranges, delete_settle  the followers: the lowest index of each group
//                  takes over the owner's outcome, the others are not found.
#include "chain_launch.h"
#include "dedup.cuh"
#include "probe.cuh"

namespace ckpp {

namespace {

constexpr int kDeleteThreads = 256;
constexpr int kDeleteWarps = kDeleteThreads / 32;
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
  uint32_t at[1];
  lists_append<1>(lists, {ws.counters + kCntFollowers}, {follows}, at);
  if (follows) write_follower(ws, at[0], i, owner);
}

template <int kTM>
__global__ void __launch_bounds__(kDeleteThreads) delete_kernel(TableSet ts, const uint8_t* __restrict__ keys,
                                                                uint64_t n, uint32_t now,
                                                                uint8_t* __restrict__ status, Workspace ws) {
  __shared__ WarpStage<1> stage[kDeleteWarps];
  __shared__ BlockLists<1> lists;
  lists_init(lists);
  pdl_wait();
  pdl_release();
  delete_chunk<kTM>(ts, keys, blockIdx.x * (uint64_t)kDeleteThreads + threadIdx.x, n, now, status, ws,
                    stage[threadIdx.x >> 5], lists);
}

// A group's lowest index takes over DELETED from its owner.
__device__ __forceinline__ void settle_range(uint8_t* __restrict__ status, const Workspace& ws, uint32_t worker,
                                             uint32_t workers) {
  const uint32_t followers = ld32_cg(ws.counters + kCntFollowers);
  for (uint32_t j = worker; j < followers; j += workers) {
    const uint2 f = ws.followers[j];
    uint8_t st = kStNotFound;
    if (f.x == ws.range[f.y].x && status[f.y] == kStDeleted) {
      st = kStDeleted;
      status[f.y] = kStNotFound;
    }
    status[f.x] = st;
  }
}

__global__ void __launch_bounds__(kSettleThreads) delete_ranges(Workspace ws) {
  pdl_wait();
  pdl_release();
  follower_ranges(ws, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(kSettleThreads) delete_settle(uint8_t* __restrict__ status, Workspace ws) {
  pdl_wait();
  pdl_release();
  settle_range(status, ws, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

}  // namespace

cudaError_t launch_delete(const TableSet& ts, const uint8_t* keys, uint64_t n, uint32_t now, uint8_t* status,
                          const Workspace& ws, cudaStream_t s) {
  const unsigned grid = grid_for(n, kDeleteThreads);
  cudaError_t e;
  if (!ts.any_timers) {
    e = launch_chained(delete_kernel<kNoTimers>, grid, kDeleteThreads, s, ts, keys, n, now, status, ws);
  } else if (!ts.views) {
    e = launch_chained(delete_kernel<kWithTimers>, grid, kDeleteThreads, s, ts, keys, n, now, status, ws);
  } else {
    e = launch_chained(delete_kernel<kTimersPerKey>, grid, kDeleteThreads, s, ts, keys, n, now, status, ws);
  }
  if (e != cudaSuccess) return e;
  const unsigned most = 2u * (unsigned)device_sm_count(), want = grid_for(n, kSettleThreads);
  const unsigned settle = want < most ? want : most;
  if ((e = launch_chained(delete_ranges, settle, kSettleThreads, s, ws)) != cudaSuccess) return e;
  return launch_chained(delete_settle, settle, kSettleThreads, s, status, ws);
}

}  // namespace ckpp
