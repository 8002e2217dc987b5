// Internal to libckpp.so: the host-side table handle and the argument and
// workspace helpers shared by the C ABI implementation files.
#pragma once

#include <cstdint>
#include <cstring>

#include "../../include/ckpp.h"
#include "ckpp_kernels.h"

struct ckpp_table {
  ckpp_geometry geo;
  uint8_t* base;
  size_t bytes;
  ckpp::TableView view;
  int have_epoch;
  uint32_t last_scan;
};

namespace ckpp {
namespace api {

constexpr size_t kAlign = 256;

constexpr size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

inline bool geometry_ok(const ckpp_geometry* g) {
  return g && g->n_buckets >= 2 && g->n_buckets <= 0xFFFFFFFFull && g->slots_per_bucket == kSlots &&
         (g->flags & ~CKPP_TIMERS) == 0;
}

inline size_t table_bytes(const ckpp_geometry* g) { return kHeaderBytes + (size_t)g->n_buckets * kBucketBytes; }

// Workspace of an n-key batch: counters | set[m] | range[n] (8 bytes each) |
// followers[n] (8) | pending[n] | retry[n] | sticky[n] (8) |
// fixup[fix_cap] (8), each part 256-byte aligned.
struct WsLayout {
  uint64_t m = 0;
  uint32_t idx_bits = 0, fix_cap = 0;
  size_t off_set = 0, off_range = 0, off_followers = 0, off_pending = 0, off_retry = 0, off_sticky = 0, off_fixup = 0,
         total = 0;
};

constexpr WsLayout ws_layout(uint64_t n) {
  WsLayout L;
  // The dedup set probes linearly, and a warp waits for the longest probe
  // sequence of its lanes (a dependent CAS per step). So m is a power of two of
  // at least 8n up to 2^17 keys (at most 4 MB of set) and 4n above (at most 2^32).
  uint64_t m = 64;
  const uint64_t want = n <= (1ull << 17) ? 8 * n : 4 * n;
  while (m < want) m <<= 1;
  L.m = m;
  while ((1ull << L.idx_bits) <= n) ++L.idx_bits;  // so that no set word equals kEmpty
  L.fix_cap = (uint32_t)(n < (1ull << 22) ? n : (1ull << 22)) + 64;
  size_t off = align_up(4 * kCounterWords, kAlign);
  L.off_set = off;
  off = align_up(off + 4 * m, kAlign);
  L.off_range = off;
  off = align_up(off + 8 * n, kAlign);
  L.off_followers = off;
  off = align_up(off + 8 * n, kAlign);
  L.off_pending = off;
  off = align_up(off + 4 * n, kAlign);
  L.off_retry = off;
  off = align_up(off + 4 * n, kAlign);
  L.off_sticky = off;
  off = align_up(off + 8 * n, kAlign);
  L.off_fixup = off;
  off = align_up(off + 8 * (size_t)L.fix_cap, kAlign);
  L.total = off;
  return L;
}

// The parts of a caller's workspace; the insert and delete launchers clear what must start at zero.
inline int carve_workspace(uint64_t n, void* workspace, size_t bytes, Workspace& ws) {
  const WsLayout L = ws_layout(n);
  if (!workspace || bytes < L.total || !aligned(workspace, kAlign)) return CKPP_EINVAL;
  uint8_t* w = static_cast<uint8_t*>(workspace);
  ws.counters = reinterpret_cast<uint32_t*>(w);
  ws.set = reinterpret_cast<uint32_t*>(w + L.off_set);
  ws.range = reinterpret_cast<uint2*>(w + L.off_range);
  ws.followers = reinterpret_cast<uint2*>(w + L.off_followers);
  ws.pending = reinterpret_cast<uint32_t*>(w + L.off_pending);
  ws.retry = reinterpret_cast<uint32_t*>(w + L.off_retry);
  ws.sticky = reinterpret_cast<unsigned long long*>(w + L.off_sticky);
  ws.fixup = reinterpret_cast<unsigned long long*>(w + L.off_fixup);
  ws.n = (uint32_t)n;
  ws.m_mask = (uint32_t)(L.m - 1);
  ws.idx_bits = L.idx_bits;
  ws.fix_cap = L.fix_cap;
  return CKPP_OK;
}

// Sec. 4.2: a timed call more than 64512 units after the last scan could see
// expired 16-bit timers wrap around and revive.
inline int time_check(ckpp_table* t, uint32_t now) {
  if (!(t->geo.flags & CKPP_TIMERS)) return CKPP_OK;
  if (!t->have_epoch) {
    t->have_epoch = 1;
    t->last_scan = now;
  }
  return (uint32_t)(now - t->last_scan) > kMaxStale ? CKPP_ESTALE : CKPP_OK;
}

inline int cuda_rc(cudaError_t e) { return e == cudaSuccess ? CKPP_OK : CKPP_ECUDA; }

// Where a buffer lives: 0 device (or managed), 1 pinned host memory mapped
// into the device's address space, -1 not reachable by the device.
inline int residency(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) return 0;
  if (a.type == cudaMemoryTypeHost && a.devicePointer == p) return 1;
  return -1;
}

// One table as a TableSet.
inline TableSet one_table(const ckpp_table* t) { return TableSet{t->view, nullptr, nullptr, 1u, t->view.timers}; }

inline int check_keys(const ckpp_key* keys, uint64_t n) {
  if (n > kMaxBatch) return CKPP_EINVAL;
  if (n && (!keys || !aligned(keys, 16))) return CKPP_EINVAL;
  return CKPP_OK;
}

}  // namespace api
}  // namespace ckpp
