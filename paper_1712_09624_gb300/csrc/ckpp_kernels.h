// Internal launchers of the GB300 Cuckoo++ kernels (host side, C++).
#pragma once

#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

#include "ckpp_device.cuh"

namespace ckpp {

// Streaming multiprocessors of the current device, queried once per device
// and cached (grid sizes of the grid-stride and persistent kernels are
// multiples of it). A failed query is not cached and returns 1, which keeps a
// grid valid; the launch that follows reports the device's error.
inline int device_sm_count() {
  constexpr int kMaxDevices = 64;
  static std::atomic<int> cache[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return 1;
  }
  int v = cache[dev].load(std::memory_order_relaxed);
  if (v > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
    cudaGetLastError();
    return 1;
  }
  cache[dev].store(v, std::memory_order_relaxed);
  return v;
}

// Words of a workspace's counters. The first 32 bytes are one sector, read at
// once where several counts are wanted, and a caller's diagnostics
// (ckpp_workspace_bytes).
constexpr uint32_t kCntPending = 0;        // keys phase 1 left (in `pending`)
constexpr uint32_t kCntFixup = 1;          // buckets whose filter may want a reset (in `fixup`)
constexpr uint32_t kCntFixupOverflow = 2;  // 1: more than `fixup` holds
constexpr uint32_t kCntMoved1 = 3;         // keys the one-move pass left (in `retry`)
constexpr uint32_t kCntFollowers = 4;      // repeated keys (in `followers`)
constexpr uint32_t kCntGrid = 5;           // keys the grid search left (in `pending`)
constexpr uint32_t kCntSecond = 6;         // keys the second search left (in `retry`)
constexpr uint32_t kCntSticky = 7;         // claimed bits to clear (in `sticky`)
constexpr uint32_t kCntRest = 8;           // blocks of the launch after a small batch's cluster that are done
constexpr uint32_t kCounterWords = 64;

// Device scratch for one insert or delete batch (carved out of the caller's
// workspace buffer, see ws_layout in api_internal.h). The counters, the set and
// the ranges are cleared before a call; every other word is written before it is
// read.
struct Workspace {
  uint32_t* counters;   // list counts (kCnt*)
  uint32_t* set;        // [m] open-addressing set of batch keys (dedup.cuh): hash bits << idx_bits | batch index of
                        // the key that claimed the position, or kEmpty
  uint2* range;         // [n] of the group that key i owns: the lowest batch index below i (kEmpty: none) and the
                        // highest above it (0: none)
  uint2* followers;     // [n] (batch index, its group's owner): the keys that repeat another key of the batch
  uint32_t* pending;    // [n] owners left for the displacement pass
  uint32_t* retry;      // [n] owners a displacement pass passes on to the next
  unsigned long long* sticky;  // [n] (batch index << 32 | bucket): buckets of timers tables whose claimed bits the
                               // finishing pass clears
  unsigned long long* fixup;   // [fix_cap] (table << 32 | bucket) whose moved counter fell to 0 off-lock
  uint32_t n;           // keys of the batch
  uint32_t m_mask;      // m - 1 (m a power of two >= 4n)
  uint32_t idx_bits;    // bits of a batch index in a set word: n < 2^idx_bits
  uint32_t fix_cap;
};

// The table(s) a mutation batch works on: one table, or many (key i goes to
// views[tab[i]]; keys naming no table are reported CKPP_ST_NO_TABLE).
struct TableSet {
  TableView single;
  const TableView* views;  // nullptr: every key goes to `single`
  const uint32_t* tab;     // per-key table index when views != nullptr
  uint32_t n_tables;
  uint32_t any_timers;     // some table has timers

  __device__ __forceinline__ bool valid(uint64_t i) const { return !views || tab[i] < n_tables; }
  __device__ __forceinline__ uint32_t id(uint64_t i) const { return views ? tab[i] : 0u; }
  __device__ __forceinline__ TableView of(uint64_t i) const { return views ? views[tab[i]] : single; }
  __device__ __forceinline__ TableView table(uint32_t id) const { return views ? views[id] : single; }
};

cudaError_t launch_init_header(uint8_t* base, uint64_t nb, uint32_t slots, uint32_t flags, uint64_t seed,
                               cudaStream_t s);

// host_io: keys and outputs are pinned host memory (read and written in place
// over NVLink-C2C). variant: 0 Cuckoo++ (filter-pruned), 1 optimistic,
// 2 pessimistic (probe.cuh).
cudaError_t launch_lookup(const TableView& t, const uint8_t* keys, uint64_t n, uint64_t* out_vals,
                          uint8_t* out_found, uint32_t now, uint32_t refresh_ttl, bool host_io, int variant,
                          cudaStream_t s);

cudaError_t launch_probe_counts(const TableView& t, const uint8_t* keys, uint64_t n, uint32_t now, int variant,
                                unsigned long long* counts, cudaStream_t s);

// Batched form (batched.cu): tables [n_tables] in device memory, jobs a device
// array of ckpp_lookup_job, n_jobs NULL or a device count (clamped to max_jobs),
// ctrl the descriptor's two zeroed counter words (chunk counter, blocks done).
cudaError_t prepare_batched_lookup();
cudaError_t launch_batched_lookup(const TableView* tables, uint32_t n_tables, const void* jobs, const uint32_t* n_jobs,
                                  uint32_t max_jobs, uint32_t now, int threads_per_key, int group_depth,
                                  int keys_per_warp, bool any_timers, uint32_t blocks, unsigned long long* ctrl,
                                  cudaStream_t s);

// Resets a carved workspace for a new batch (clear_workspace in dedup.cuh) in one
// launch.
cudaError_t launch_workspace_clear(const Workspace& ws, cudaStream_t s);

// The insert launch modes a caller can pick (insert.cu).
constexpr int kInsertLaunchChain = 0, kInsertLaunchSingle = 1;
int set_insert_launch(int mode);  // returns the previous mode, or -1 for an unknown mode

cudaError_t launch_insert(const TableSet& ts, const uint8_t* keys, const uint64_t* vals, uint64_t n,
                          uint32_t now, uint32_t expiry, uint8_t* status, const Workspace& ws, cudaStream_t s);

cudaError_t launch_delete(const TableSet& ts, const uint8_t* keys, uint64_t n, uint32_t now, uint8_t* status,
                          const Workspace& ws, cudaStream_t s);

cudaError_t launch_expire(const TableView& t, uint32_t now, unsigned long long* n_expired, cudaStream_t s);

// out: 7 sums + 16 histogram bins (uint64), zeroed by the caller.
cudaError_t launch_stats(const TableView& t, uint32_t now, unsigned long long* out, cudaStream_t s);

}  // namespace ckpp
