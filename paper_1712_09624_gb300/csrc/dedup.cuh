// In-batch duplicate keys of an insert or delete call. A batch has the result
// of applying its keys one by one in index order, but equal keys are found
// while the batch runs: an open-addressing set in the workspace gives each
// group of equal keys one owner, the member that claims the group's position
// first, whichever that is. The owner does the group's work on the table; the
// other members (followers) are listed and widen the group's range of batch
// indices, and the call's last kernel settles the group: the lowest index
// reports the outcome, the others that of a repeated key, and an insert stores
// the value of the highest index.
// So a key that occurs once (nearly all of them) pays for one CAS, which its
// owner issues together with the read of its bucket, and no later pass looks
// at it. (A separate dedup kernel before the table kernels, with a claimed
// position's first and last index side by side and a flag byte per key, took
// 28 us of a 1M-key call and as much again in reads by the passes after it.)
//
// A set word is 4 bytes: the batch index in its low idx_bits and as many hash
// bits as remain above it, so that a position held by another key is passed over
// without reading that key (1M keys: 11 bits, one false match in 2048).
// Position and word come from a hash of their own, its upper and its lower half.
// The keys of a batch may share any part of their primary hash: a shard's keys
// share bits 16-31 of it, keys of a few buckets its upper bits. (Taken from the
// primary hash itself, the position from bit 16 on, 1M keys of one shard of eight
// passed 4,097 positions each where they pass 0.17 now; and a word's bits were a
// part of its position, so that 99 % of the keys met were read.)
#pragma once

#include "mutate.cuh"

namespace ckpp {

constexpr uint32_t kWarpAll = 0xFFFFFFFFu;
constexpr uint32_t kNoIndex = 0xFFFFFFFFu;

__device__ __forceinline__ Key load_key(const uint8_t* keys, uint64_t i) { return ld_key(keys + 16 * i); }
// As ld_key, not by the read-only path.
__device__ __forceinline__ uint64_t load_val(const uint64_t* vals, uint64_t i) {
  uint64_t v;
  asm volatile("ld.global.u64 %0, [%1];" : "=l"(v) : "l"(vals + i) : "memory");
  return v;
}

// A key's probe of the set: its position, its word and what the CAS returned.
struct SetProbe {
  uint32_t pos, word, old;
};

// The first CAS (h1: the key's primary hash, tid: its table). Its result is
// not looked at here, so that the caller can request more before waiting.
__device__ __forceinline__ SetProbe set_probe(const Workspace& ws, uint64_t h1, uint32_t tid, uint32_t i) {
  const uint64_t h = mix64(h1 ^ (uint64_t)tid * 0x9E3779B97F4A7C15ull);  // one key bound for many tables spreads out
  SetProbe p;
  p.pos = (uint32_t)(h >> 32) & ws.m_mask;
  p.word = ((uint32_t)h >> ws.idx_bits << ws.idx_bits) | i;
  p.old = atomicCAS(ws.set + p.pos, kEmpty, p.word);
  return p;
}

// The owner of key i's group: i itself if a probe found a free position (the
// set has 4n positions or more, so one is met). Equal keys bound for
// different tables are different keys.
__device__ __forceinline__ uint32_t set_owner(const Workspace& ws, const TableSet& ts, const uint8_t* keys,
                                              const Key& k, uint32_t tid, uint32_t i, SetProbe p) {
  for (uint32_t n = 0; n <= ws.m_mask; ++n) {
    if (p.old == kEmpty) return i;
    if (((p.old ^ p.word) >> ws.idx_bits) == 0u) {
      const uint32_t cur = p.old & ((1u << ws.idx_bits) - 1u);
      const Key o = load_key(keys, cur);
      if (o.k0 == k.k0 && o.k1 == k.k1 && ts.id(cur) == tid) return cur;
    }
    p.pos = (p.pos + 1) & ws.m_mask;
    p.old = atomicCAS(ws.set + p.pos, kEmpty, p.word);
  }
  return i;
}

// Appending to lists. Every returning atomic on one counter, or on two counters
// of one 128-byte line, takes 0.8 ns (a warp's append to one list each, of a
// 1M-key batch: 26 us), so a block takes its places with one atomic per list.
template <int kLists>
struct BlockLists {
  uint32_t count[kLists], base[kLists];
};

// Before the first append (block-wide).
template <int kLists>
__device__ __forceinline__ void lists_init(BlockLists<kLists>& L) {
  if (threadIdx.x < kLists) L.count[threadIdx.x] = 0;
  __syncthreads();
}

// at[j] receives this thread's place in list j where want[j] (block-wide: every
// thread of the block calls this).
template <int kLists>
__device__ __forceinline__ void lists_append(BlockLists<kLists>& L, uint32_t* const (&counters)[kLists],
                                             const bool (&want)[kLists], uint32_t (&at)[kLists]) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int j = 0; j < kLists; ++j) {
    const uint32_t mask = __ballot_sync(kWarpAll, want[j]);
    at[j] = 0;
    if (mask) {
      const uint32_t leader = __ffs(mask) - 1;
      uint32_t first = 0;
      if (lane == leader) first = atomicAdd(&L.count[j], (uint32_t)__popc(mask));
      at[j] = __shfl_sync(kWarpAll, first, leader) + __popc(mask & ((1u << lane) - 1u));
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kLists; ++j) {
    if (threadIdx.x == 32 * j && L.count[j]) {
      L.base[j] = atomicAdd(counters[j], L.count[j]);
      L.count[j] = 0;
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kLists; ++j)
    if (want[j]) at[j] += L.base[j];
}

// Key i as a follower of owner, at place at of the list; its group's range is
// widened to include it. (The range is widened here and not by a kernel after the
// owners', which cost a launch or a barrier: a delete of 8K absent keys 12.4 ->
// 10.4 us, insert and delete of 4K to 8K keys 2 us less; its price is the clear of
// 8 bytes per key, and 6 us of 67 where 90 % of 128K keys are repeated.)
__device__ __forceinline__ void write_follower(const Workspace& ws, uint32_t at, uint32_t i, uint32_t owner) {
  ws.followers[at] = make_uint2(i, owner);
  if (i < owner) {
    atomicMin(&ws.range[owner].x, i);
  } else {
    atomicMax(&ws.range[owner].y, i);
  }
}

// All counts at once.
struct Counts {
  uint32_t c[8];
  __device__ __forceinline__ uint32_t operator[](uint32_t i) const { return c[i]; }
};

__device__ __forceinline__ Counts load_counts(const Workspace& ws) {
  uint64_t w[4];
  ld256_cg(ws.counters, w);
  Counts r;
#pragma unroll
  for (int i = 0; i < 8; ++i) r.c[i] = (uint32_t)(w[i / 2] >> (32 * (i & 1)));
  return r;
}

// The workspace of a call that one block runs alone (at most kOneBlockKeys
// keys), its set, ranges and followers moved to shared memory.
constexpr uint32_t kOneBlockKeys = 256;
struct OneBlockSet {
  __align__(16) uint32_t set[8 * kOneBlockKeys];
};
struct OneBlockGroups {
  __align__(16) uint2 range[kOneBlockKeys];
  uint2 followers[kOneBlockKeys];
};
__device__ __forceinline__ Workspace in_shared(Workspace ws, OneBlockSet& set, OneBlockGroups& groups) {
  ws.set = set.set;
  ws.range = groups.range;
  ws.followers = groups.followers;
  return ws;
}

// Reset the counters to 0, the set to empty and the ranges to none. (m is a
// power of two >= 64, and the set and the ranges are parts of their own, 256-byte
// aligned: whole 16-byte vectors.)
__device__ __forceinline__ void clear_workspace(const Workspace& ws, uint32_t worker, uint32_t workers) {
  uint4* set = reinterpret_cast<uint4*>(ws.set);
  const uint64_t n_vec = ((uint64_t)ws.m_mask + 1) / 4;
  for (uint32_t j = worker; j < kCounterWords; j += workers) ws.counters[j] = 0u;
  for (uint64_t j = worker; j < n_vec; j += workers) set[j] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
  uint4* range = reinterpret_cast<uint4*>(ws.range);
  for (uint32_t j = worker; j < (ws.n + 1) / 2; j += workers) range[j] = make_uint4(kEmpty, 0u, kEmpty, 0u);
}

// All threads of the cluster arrive; what each wrote before is seen by all after.
// Not the .aligned forms: those want every warp whole at the barrier, and lanes
// come to it from loops and lock waits of different lengths.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

}  // namespace ckpp
