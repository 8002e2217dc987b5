// Bulk lookup over one table (Sec. 2 and Sec. 4.1 of the paper): each warp
// takes 32 keys, one per lane, and fetches their bucket lines together into
// shared memory (probe.cuh).
//
// The paper hides DRAM latency by interleaving the steps of a batch of lookups
// with prefetches (Sec. 3); on the GPU the same memory-level parallelism comes
// from every warp keeping its 32 keys' line requests in flight at once, over
// the tens of warps resident on each SM. Blocks are short-lived and launched in
// key order, so at any time the resident warps read keys, and write results,
// within one narrow window of the batch. (Measured: warps that each walk a long
// span of the batch, with their next keys prefetched, ran 10-20% slower.)
// Keys are read with coalesced 16-byte loads and results written with
// coalesced stores.
#include "chain_launch.h"
#include "probe.cuh"

namespace ckpp {

namespace {

constexpr int kLookupThreads = 128;  // 4 warps: 17 KB of line slabs per block
constexpr int kWarpsPerBlock = kLookupThreads / 32;

// kHostIO: keys and results live in pinned host memory, reached over
// NVLink-C2C by the loads and stores themselves (no staging copy); such keys
// are read with plain loads, without cache hints, and each
// warp writes its results as 16-byte vectors (small scattered stores are what
// the link does worst) when the output pointers allow it.
// kCount: no results; the secondary-line, record and second-line reads are
// added to counts[1..3] and the keys to counts[0].
template <bool kCount, bool kHostIO, int kVariant, int kTM>
__global__ void __launch_bounds__(kLookupThreads) lookup_kernel(TableView t, const uint8_t* __restrict__ keys,
                                                                uint64_t n, uint64_t* __restrict__ out_vals,
                                                                uint8_t* __restrict__ out_found, uint32_t now,
                                                                uint32_t refresh_ttl,
                                                                unsigned long long* __restrict__ counts) {
  __shared__ WarpStage<1> stage[kWarpsPerBlock];
  __shared__ __align__(16) uint64_t vals[kHostIO ? kLookupThreads : 1];
  __shared__ __align__(16) uint8_t flags[kHostIO ? kLookupThreads : 1];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t c = (uint64_t)blockIdx.x * kWarpsPerBlock + warp;  // the warp's 32-key chunk
  const uint64_t i = c * 32 + lane;
  pdl_wait();
  bool act[1] = {i < n};
  Key k{0, 0};
  if (act[0]) {
    k = kHostIO ? ld_key(keys + 16 * i) : ld_key_stream(keys + 16 * i, policy_evict_first());
  }
  Probe p[1];
  probe_init(p[0], k, t.buckets, t.nb, t.seed, t.timers);
  run_probes<kVariant, kCount, 1, kTM>(p, act, now, stage[warp]);
  if (kCount) {
    const uint32_t nkey = __reduce_add_sync(kFull, act[0] ? 1u : 0u);
    const uint32_t nsec = __reduce_add_sync(kFull, p[0].nsec);
    const uint32_t nrec = __reduce_add_sync(kFull, p[0].nrec);
    const uint32_t nl1 = __reduce_add_sync(kFull, p[0].nline1);
    if (lane == 0 && nkey) {
      atomicAdd(counts + 0, (unsigned long long)nkey);
      atomicAdd(counts + 1, (unsigned long long)nsec);
      atomicAdd(counts + 2, (unsigned long long)nrec);
      atomicAdd(counts + 3, (unsigned long long)nl1);
    }
    return;
  }
  // Sec. 4.2: a hit may refresh the entry's expiry.
  if (kTM == kWithTimers && act[0] && p[0].found && refresh_ttl) set_expiry(t, p[0].hb, p[0].hs, now + refresh_ttl);
  const bool vec = kHostIO && (reinterpret_cast<uintptr_t>(out_vals) % 16 == 0) &&
                   (reinterpret_cast<uintptr_t>(out_found) % 16 == 0);
  if (vec && c * 32 + 32 <= n) {
    uint64_t* wv = vals + warp * 32;
    uint8_t* wf = flags + warp * 32;
    wv[lane] = p[0].value;
    wf[lane] = p[0].found ? 1 : 0;
    __syncwarp();
    if (lane < 16) {
      reinterpret_cast<ulonglong2*>(out_vals + c * 32)[lane] = reinterpret_cast<const ulonglong2*>(wv)[lane];
    } else if (lane < 18) {
      reinterpret_cast<uint4*>(out_found + c * 32)[lane - 16] = reinterpret_cast<const uint4*>(wf)[lane - 16];
    }
  } else if (act[0]) {
    out_vals[i] = p[0].value;
    out_found[i] = p[0].found ? 1 : 0;
  }
}

// The lookup of a table that (mostly) stays in L2, one thread per key without
// staging: the bucket's header is read with one 32-byte load, and only a slot
// whose tag matches costs more (its key, value and expiry, requested
// together). On a table beyond L2 each of these reads is a random DRAM access
// of its own, which is why lookup_kernel fetches whole lines; in L2 they run at
// 250 G/s, and lookup_kernel is bound by its 22 warp instructions per lookup
// instead. 1M keys, half of them unknown, load 0.9: 26.8 -> 14.4 us on a 32 MB
// table (28.8 -> 18.8 when three such tables take turns, 16.1 since calls are
// chained). Blocks of 128 threads: 15.7, of 64 and 256 16.1, of 512 16.7.
constexpr int kDirectThreads = 128;

template <int kTM>
__global__ void __launch_bounds__(kDirectThreads) lookup_direct_kernel(TableView t, const uint8_t* __restrict__ keys,
                                                                       uint64_t n, uint64_t* __restrict__ out_vals,
                                                                       uint8_t* __restrict__ out_found, uint32_t now) {
  constexpr uint32_t timers = kTM == kWithTimers ? 1u : 0u;
  const uint64_t i = blockIdx.x * (uint64_t)kDirectThreads + threadIdx.x;
  pdl_wait();
  if (i >= n) return;
  const Key k = ld_key_stream(keys + 16 * i, policy_evict_first());
  const uint64_t h1 = hash_key(k, t.seed);
  const uint32_t tag = (uint32_t)(h1 & 0xFFFF);
  uint32_t b = reduce(h1, t.nb);
  bool found = false;
  uint64_t value = 0;
  for (int which = 0;; ++which) {
    uint64_t h[4];
    const uint8_t* bucket = bucket_ptr(t, b);
    ld256_cg(bucket, h);
    const uint4 tags = make_uint4((uint32_t)h[0], (uint32_t)(h[0] >> 32), (uint32_t)h[1], (uint32_t)(h[1] >> 32));
    uint32_t cand = tag_mask16(tags, tag) & (uint32_t)h[3] & kBusyMask;
    bool stored = false;
    while (cand) {
      const uint32_t s = __ffs(cand) - 1;
      cand &= cand - 1;
      uint64_t k0, k1;
      ld128_cg(bucket + key_off(timers, s), k0, k1);
      const uint64_t v = ld64_cg(bucket + value_off(timers, s));
      const uint32_t e = timers ? ld16_cg(bucket + kExpiryOff + 2u * s) : 0u;
      if (k0 == k.k0 && k1 == k.k1) {
        stored = true;
        if (!timers || alive16(e, now)) {  // Sec. 4.2: a dead entry is not returned
          found = true;
          value = v;
        }
        break;
      }
    }
    if (stored || which) break;
    // Sec. 4.1: the secondary only if both of the key's bits are set in the primary's filter
    const uint64_t h2 = hash_key(k, t.seed ^ kSeed2Xor);
    const uint64_t bits = (1ull << (h2 & 63)) | (1ull << ((h2 >> 6) & 63));
    if ((h[2] & bits) != bits) break;
    const uint32_t b2 = reduce(h2, t.nb);
    b = b2 != b ? b2 : (b + 1 == (uint32_t)t.nb ? 0u : b + 1);
  }
  out_vals[i] = value;
  out_found[i] = found ? 1 : 0;
}

// Largest table (bytes of buckets) that lookup_direct_kernel is used for: one
// whose first lines, half of it, fit in L2. Its reads are sectors of one line,
// but each its own DRAM access once the line has gone. 4M keys, all known, load
// 0.3 / 0.5 / 0.9, lookup_kernel -> this one in us: 240 MB 78 -> 61 / 90 -> 68 /
// 116 -> 101 (with timers 96 -> 76 / 108 -> 83 / 137 -> 111), 248 MB 79 -> 89 /
// 90 -> 97 / 117 -> 102, 256 MB 79 -> 100 / 90 -> 103 / 117 -> 104 (with timers
// 96 -> 132 / 110 -> 131 / 139 -> 114). Tables that take turns, 512 MB or more
// in all, gain as much up to 240 MB each. A lookup that refreshes its hits keeps
// to lookup_kernel: the refresh's store follows three reads of the bucket instead
// of one (32 MB, load 0.6, all known: 30.8 us there, 35.1 here).
constexpr uint64_t kDirectBytes = 240ull << 20;

cudaError_t launch_direct(const TableView& t, const uint8_t* keys, uint64_t n, uint64_t* out_vals, uint8_t* out_found,
                          uint32_t now, cudaStream_t s) {
  const uint64_t blocks = (n + kDirectThreads - 1) / kDirectThreads;
  return launch_chained(t.timers ? lookup_direct_kernel<kWithTimers> : lookup_direct_kernel<kNoTimers>, (unsigned)blocks,
                        kDirectThreads, s, t, keys, n, out_vals, out_found, now);
}

template <bool kCount, bool kHostIO, int kVariant>
cudaError_t launch(const TableView& t, const uint8_t* keys, uint64_t n, uint64_t* out_vals, uint8_t* out_found,
                   uint32_t now, uint32_t refresh_ttl, unsigned long long* counts, cudaStream_t s) {
  const uint64_t blocks = ((n + 31) / 32 + kWarpsPerBlock - 1) / kWarpsPerBlock;
  return launch_chained(t.timers ? lookup_kernel<kCount, kHostIO, kVariant, kWithTimers>
                                 : lookup_kernel<kCount, kHostIO, kVariant, kNoTimers>,
                        (unsigned)blocks, kLookupThreads, s, t, keys, n, out_vals, out_found, now,
                        t.timers ? refresh_ttl : 0u, counts);
}

}  // namespace

cudaError_t launch_lookup(const TableView& t, const uint8_t* keys, uint64_t n, uint64_t* out_vals,
                          uint8_t* out_found, uint32_t now, uint32_t refresh_ttl, bool host_io, int variant,
                          cudaStream_t s) {
  if (host_io) {
    if (variant != kBloom) return cudaErrorInvalidValue;
    return launch<false, true, kBloom>(t, keys, n, out_vals, out_found, now, refresh_ttl, nullptr, s);
  }
  if (variant == kBloom && !refresh_ttl && t.nb * kBucketBytes <= kDirectBytes)
    return launch_direct(t, keys, n, out_vals, out_found, now, s);
  switch (variant) {
    case kBloom: return launch<false, false, kBloom>(t, keys, n, out_vals, out_found, now, refresh_ttl, nullptr, s);
    case kOptimistic:
      return launch<false, false, kOptimistic>(t, keys, n, out_vals, out_found, now, refresh_ttl, nullptr, s);
    case kPessimistic:
      return launch<false, false, kPessimistic>(t, keys, n, out_vals, out_found, now, refresh_ttl, nullptr, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_probe_counts(const TableView& t, const uint8_t* keys, uint64_t n, uint32_t now, int variant,
                                unsigned long long* counts, cudaStream_t s) {
  switch (variant) {
    case kBloom: return launch<true, false, kBloom>(t, keys, n, nullptr, nullptr, now, 0, counts, s);
    case kOptimistic: return launch<true, false, kOptimistic>(t, keys, n, nullptr, nullptr, now, 0, counts, s);
    case kPessimistic: return launch<true, false, kPessimistic>(t, keys, n, nullptr, nullptr, now, 0, counts, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ckpp
