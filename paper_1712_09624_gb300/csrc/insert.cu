// Batched insert-or-update (Sec. 2 cuckoo insertion; Sec. 4.1 filter and moved
// counter upkeep; Sec. 4.2 reuse of dead slots).
//
// Kernels, in stream order:
//   phase1  - per key, lock-free: the duplicate-key set (dedup.cuh) gives each
//             group of equal keys one owner, which updates the key in place if
//             it is stored (a dead entry is revived), else claims the lowest
//             free or dead slot of the primary, else of the secondary, with a
//             CAS on the bucket's ctrl word, writes the entry into the claimed
//             slot and publishes it; owners with two full buckets are queued
//             for the displacement passes.
//   move1   - per queued owner: the cuckoo paths of length one. Read the
//             entries of b1, then of b2, and the buckets they can move to; the
//             first entry whose other bucket has a free or dead slot moves
//             there under the locks of the path, and the key takes its slot.
//             At load factor 0.9 it places nearly every queued key.
//   phase2  - per key move1 left: breadth-first search for a longer cuckoo
//             path without locks (queue in shared memory), then lock every
//             bucket of the path plus the key's primary, re-validate the path,
//             and move the entries backwards and store the key, all under
//             those locks; retry a bounded number of times. One thread per
//             key, or one warp per key for a short list. Keys still
//             unplaced get a wider search, then the widest, each run by a
//             whole warp per key (a level of the search in two round trips);
//             only then FULL.
//   fixup and finish (one kernel) - reset the filter of buckets whose moved
//             counter reached zero off their lock (the reset of Sec. 4.1,
//             deferred so that it never races a concurrent setter), clear the
//             claimed bits that phase 1 left set in timers tables, and settle
//             the groups of equal keys (the first occurrence reports the
//             outcome, later ones UPDATED, or FULL/BUSY; the last one's value
//             is stored), which gives the batch the result of inserting its
//             keys one by one in index order.
// Before them, one kernel clears the workspace (counters, set and ranges). Each
// kernel waits for its predecessor in its first instruction (chain_launch.h).
#include "chain_launch.h"
#include "dedup.cuh"

namespace ckpp {

namespace {

constexpr int kThreads = 256;
constexpr int kPathAttempts = 16;
// Buckets the one-move pass reads per round trip when looking for room for a root's entries.
constexpr uint32_t kMoveGroup = 2;

// --------------------------------------------------------------- phase 1
// Per key, without locks: the duplicate-key set (dedup.cuh) decides whether it
// owns its group; an owner then finds its key or a slot for it.
//
// A key that is stored (alive or dead, Sec. 4.2) is found in its primary
// bucket, or in its secondary when the primary's filter says it may be there
// (Sec. 4.1: a key stored in its secondary has both bits set in its primary's
// filter; phase 1 moves no entry and each key has one owner, so the tests are
// exact). A live entry is updated in place. Any other key claims the lowest
// claimable slot of its primary, else of its secondary (Sec. 2), else waits
// for the displacement passes.
//
// A claim is a CAS on the bucket's ctrl word that sets the slot's claimed bit.
// A failed CAS returns the current word, and the claimable slots are recomputed
// from it. The owner then writes the entry. A slot that was free is published
// after a fence by one atomic XOR, which turns the claimed bit into busy:
// readers look at busy slots only, and one that meets a busy slot with its
// key's tag reads the slot's key behind a fence of its own, so it never sees
// the bytes that a freshly published slot held before.
//
// A slot that holds a dead entry (timers) stays busy when it is claimed (the
// dead entry is evicted, with moved-counter upkeep on its own primary; the
// in_secondary bit becomes the new entry's) and keeps its claimed bit until the
// finishing pass (listed in ws.sticky): it needs no publication, readers pass
// over claimed slots, and its word never reads again as it did before the
// claim. Reviving a key's own dead entry claims its slot in the same way, so a
// revival and a reuse of that slot by another key cannot both succeed. And a
// slot counts as dead only if its expiry was read after (a fence) the ctrl word
// that showed it busy.
//
// Storing a key in its secondary sets its two bits in the primary's filter and
// counts it in the primary's moved counter, with relaxed atomics: no filter is
// reset during phase 1 (resets of counters that reach zero here are deferred
// to the finishing pass). Nothing in phase 1 waits on another thread.
//
// What bounds it is the number of line requests, reads, writes and atomics
// alike: on a 4 GiB buffer a thread per random line runs at 47 G/s with one
// 32-byte read, at 24 with a store to the line after it, at 12 with three, and
// at 8 with the whole sequence of a claim made by one thread (read, CAS, stores
// of key, value and tag, XOR). Lanes that touch one line in one instruction
// make one request together, so a warp gathers its keys' work: with timers the
// header and the expiries come with one request (p1_fetch), and an entry's key
// and value go out with one, its tag and expiry with another (p1_store).
// Whole insert calls against separate dedup, claim and publication kernels that
// made every request lane by lane: 1M keys into 134M slots at load 0.8 275 ->
// 205 us, into 34M slots at 0.5 245 -> 175 us, with timers 280 -> 183 us; 64K
// keys at 0.8 72 -> 65 us. (Taking exclusive ownership of a key's buckets in the
// L2-resident set first, so that the table needs no atomics, was measured too:
// 212 us where this takes 205, and slower with timers or with many keys per
// bucket; the claims in the set cost what they save on the table.)
constexpr int kClaimAttempts = 64;  // CAS retries on one bucket (two changes of its word per slot at most)

__device__ __forceinline__ uint32_t claim_bit(uint32_t s) { return 1u << (kClaimShift + s); }

// The slots that phase 1 may claim in a bucket whose word is c: free, or in
// dead (busy slots found dead), and not claimed.
__device__ __forceinline__ uint32_t claimable(uint32_t c, uint32_t dead) {
  return (~c | dead) & ~(c >> kClaimShift) & kBusyMask;
}

// A warp's rows in shared memory: the first 64 bytes of a bucket each, or a
// store job each. 16-byte chunk c of row r is kept at c ^ (r >> 1 & 3).
struct P1Rows {
  unsigned long long addr[32];
  __align__(128) uint4 row[32][4];
};
__device__ __forceinline__ uint4& row_chunk(P1Rows& R, uint32_t r, uint32_t c) { return R.row[r][c ^ ((r >> 1) & 3u)]; }

// A bucket as phase 1 sees it.
struct P1Bucket {
  uint32_t b, ctrl, match;  // match: busy slots with the key's tag that no key has claimed
  uint32_t dead;            // busy slots with a dead entry (timers)
  uint32_t fresh;           // slots with the expiry that this batch writes (timers; only where match is set)
  uint64_t bloom;
};

// Which of r's slots are dead and which carry the batch's own expiry, from one
// reading of the expiries (e0, e1): another key's expiry that makes a dead slot
// look alive always shows in fresh as well.
__device__ __forceinline__ void p1_expiries(P1Bucket& r, uint64_t e0, uint64_t e1, uint32_t now, uint32_t expiry) {
  r.dead = r.ctrl & ~alive_mask(e0, e1, now) & kBusyMask;
  r.fresh = r.match ? tag_mask(e0, e1, expiry) : 0u;
}

// From one reading, in no order: dead and match may name slots that another key
// has taken or published meanwhile, until p1_search.
__device__ __forceinline__ P1Bucket p1_bucket(uint32_t b, const Snap& s, uint32_t tag, bool timers, uint32_t now,
                                              uint32_t expiry) {
  P1Bucket r;
  r.b = b;
  r.ctrl = (uint32_t)s.w[3];
  r.match = tag_mask(s.w[0], s.w[1], tag) & r.ctrl & ~(r.ctrl >> kClaimShift) & kBusyMask;
  r.bloom = s.w[2];
  r.dead = r.fresh = 0;
  if (timers) p1_expiries(r, s.e0, s.e1, now, expiry);
  return r;
}

// The header and (timers) the expiries of bucket b for every lane that wants
// one (the whole warp calls this). With timers four lanes copy a bucket's first
// 64 bytes together: reading them with two loads per lane is two requests.
template <bool kTimers>
__device__ __forceinline__ void p1_fetch(const TableView& t, uint32_t b, bool want, P1Rows& R, Snap& s) {
  if (!kTimers) {
    if (want) ld256_cg(bucket_ptr(t, b), s.w);
    return;
  }
  const uint32_t lane = threadIdx.x & 31u, mask = __ballot_sync(kWarpAll, want);
  if (!mask) return;
  const uint32_t rank = __popc(mask & ((1u << lane) - 1u)), n = __popc(mask);
  if (want) R.addr[rank] = reinterpret_cast<unsigned long long>(bucket_ptr(t, b));
  __syncwarp();
  for (uint32_t j = lane >> 2; j < n; j += 8) {
    const uint32_t c = lane & 3u;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&row_chunk(R, j, c));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(R.addr[j] + 16u * c) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  if (want) {
    const uint4 a = row_chunk(R, rank, 0), h = row_chunk(R, rank, 1), e = row_chunk(R, rank, kExpiryOff / 16u);
    s.w[0] = lo64(a), s.w[1] = hi64(a), s.w[2] = lo64(h), s.w[3] = hi64(h);
    s.e0 = lo64(e), s.e1 = hi64(e);
  }
  __syncwarp();
}

// The same for one lane (rare).
__device__ __forceinline__ void p1_fetch_one(const TableView& t, uint32_t b, bool timers, Snap& s) {
  ld256_cg(bucket_ptr(t, b), s.w);
  s.e0 = s.e1 = 0;
  if (timers) ld128_cg(expiry_ptr(t, b, 0), s.e0, s.e1);
}

// The slot of bucket r holding key k, or -1 (behind a fence that follows r).
__device__ __forceinline__ int p1_find(const TableView& t, const P1Bucket& r, const Key& k) {
  uint32_t cand = r.match;
  while (cand) {
    const int slot = __ffs(cand) - 1;
    cand &= cand - 1;
    uint64_t k0, k1;
    ld128_cg(key_ptr(t, r.b, slot), k0, k1);
    if (k0 == k.k0 && k1 == k.k1) return slot;
  }
  return -1;
}

// What has to be read behind the ctrl words of the primary r and of the
// secondary r2 (empty if it was not read): the expiries again, where they showed
// a dead slot, and the keys of the slots that match. Returns the slot of key k,
// in r2 if second, or -1. One fence and one round trip serve both buckets (a
// fence for each reading, up to four in a row: an insert of 1M keys of an
// 8M-slot table full of dead entries, half of them revived, 183 -> 162 us).
__device__ __forceinline__ int p1_search(const TableView& t, P1Bucket& r, P1Bucket& r2, const Key& k, uint32_t now,
                                         uint32_t expiry, bool& second) {
  second = false;
  if (!(r.match | r.dead | r2.match | r2.dead)) return -1;
  fence_acq_rel();
  uint64_t e0 = 0, e1 = 0, f0 = 0, f1 = 0;
  if (r.dead) ld128_cg(expiry_ptr(t, r.b, 0), e0, e1);
  if (r2.dead) ld128_cg(expiry_ptr(t, r2.b, 0), f0, f1);
  int slot = p1_find(t, r, k);
  if (slot < 0) {
    slot = p1_find(t, r2, k);
    second = slot >= 0;
  }
  if (r.dead) p1_expiries(r, e0, e1, now, expiry);
  if (r2.dead) p1_expiries(r2, f0, f1, now, expiry);
  return slot;
}

// Claim the slot of the key's own dead entry (slot sl of bucket b, busy in c).
// Returns 1 on success, 0 if another key took the slot first (the entry is
// gone), -2 (latched) after kClaimAttempts failed CASes.
__device__ int claim_revival(const TableView& t, uint32_t b, uint32_t sl, uint32_t c) {
  uint32_t* cp = ctrl_ptr(t, b);
  for (int i = 0; i < kClaimAttempts; ++i) {
    if (!((c >> sl) & 1u) || ((c >> (kClaimShift + sl)) & 1u)) return 0;
    const uint32_t got = atomicCAS(cp, c, c | claim_bit(sl));
    if (got == c) return 1;
    c = got;
  }
  latch_error(t, kErrLockTimeout);
  return -2;
}

// What a key does with its slot.
enum P1Work : uint32_t { kP1None, kP1Update, kP1Revive, kP1Place };

// The key is stored in slot sl of bucket r: a live entry is updated in place
// (UPDATED), a dead one revived through a claim (INSERTED, Sec. 4.2). Returns
// the status, or 0 if the entry turned out to be a dead one that another key
// has just taken.
__device__ __forceinline__ uint8_t p1_stored(const TableView& t, const P1Bucket& r, uint32_t sl, bool timers,
                                             P1Work& work) {
  work = kP1Update;
  if (timers) {
    if ((r.dead >> sl) & 1u) {
      const int got = claim_revival(t, r.b, sl, r.ctrl);
      work = got > 0 ? kP1Revive : kP1None;
      return got > 0 ? kStInserted : got == 0 ? 0 : kStBusy;
    }
    // The expiry that called the entry alive may be that of a key of this batch which
    // has taken the slot since its word was read: then the word shows the claim by now.
    if ((r.fresh >> sl) & 1u) {
      fence_acq_rel();
      if ((ld32_cg(ctrl_ptr(t, r.b)) >> (kClaimShift + sl)) & 1u) {
        work = kP1None;
        return 0;
      }
    }
  }
  return kStUpdated;
}

// Claim the lowest claimable slot of bucket r (insec: the key's secondary).
// Returns the slot (prev receives the word the CAS replaced), -1 if nothing is
// claimable, -2 (latched) after kClaimAttempts failed CASes.
__device__ __forceinline__ int claim_slot(const TableView& t, const P1Bucket& r, bool insec, uint32_t& prev) {
  uint32_t* cp = ctrl_ptr(t, r.b);
  uint32_t c = r.ctrl;
  for (int i = 0; i < kClaimAttempts; ++i) {
    const uint32_t f = claimable(c, r.dead);
    if (!f) return -1;
    const uint32_t sl = __ffs(f) - 1;
    const uint32_t in = 1u << (kInsecShift + sl);
    const uint32_t want = ((c | claim_bit(sl)) & ~in) | (insec && ((c >> sl) & 1u) ? in : 0u);
    const uint32_t got = atomicCAS(cp, c, want);
    if (got == c) {
      prev = c;
      return (int)sl;
    }
    c = got;
  }
  latch_error(t, kErrLockTimeout);
  return -2;
}

// Store the warp's nj jobs. Row j of R: the key; the value and the bucket's
// address; then which words to write (bits 0-5: the key's and the value's
// four-byte words, 6 the tag, 7 the expiry) | slot << 8 | timers << 16, and
// tag | expiry << 16. Six lanes store a job's key and value, two more its tag
// and expiry in a second instruction (their neighbours belong to other keys'
// claims, so they go out as 16-bit words).
template <bool kTimers>
__device__ __forceinline__ void p1_store(uint32_t nj, P1Rows& R) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t q = lane / 6u, c = lane % 6u;
  for (uint32_t j = q < 5u ? q : nj; j < nj; j += 5) {
    const uint4 what = row_chunk(R, j, 2);
    const uint4 vb = row_chunk(R, j, 1);
    if (!((what.x >> c) & 1u)) continue;
    const uint32_t s = (what.x >> 8) & 7u, timers = kTimers ? what.x >> 16 : 0u;
    const uint32_t w = c < 4u ? reinterpret_cast<const uint32_t*>(&row_chunk(R, j, 0))[c] : (c == 4u ? vb.x : vb.y);
    const uint32_t off = c < 4u ? key_off(timers, s) + 4u * c : value_off(timers, s) + 4u * (c - 4u);
    *reinterpret_cast<uint32_t*>(hi64(vb) + off) = w;
  }
  const uint32_t half = lane & 1u;
  for (uint32_t j = lane >> 1; j < nj; j += 16) {
    const uint4 what = row_chunk(R, j, 2);
    if (!((what.x >> (6u + half)) & 1u)) continue;
    const uint32_t off = 2u * ((what.x >> 8) & 7u) + (half ? kExpiryOff : 0u);
    *reinterpret_cast<uint16_t*>(hi64(row_chunk(R, j, 1)) + off) = (uint16_t)(half ? what.y >> 16 : what.y);
  }
}

// The lists a thread appends to in phase 1: displacement passes, followers, sticky.
using P1Lists = BlockLists<3>;

// One key of phase 1 (every thread of the block calls this; act: it has a
// key). A warp takes the steps of all its keys together, so its lanes' memory
// round trips overlap: the key; the set's CAS and the primary's header; the
// secondary's header, for the keys whose filter bits are set or whose primary
// has no room; the claim; the entry; the publication.
template <bool kTimers>
__device__ __forceinline__ void phase1_one(const TableSet& ts, const uint8_t* __restrict__ keys,
                                           const uint64_t* __restrict__ vals, uint32_t now, uint32_t expiry,
                                           uint8_t* __restrict__ status, const Workspace& ws, uint64_t i64, bool act,
                                           P1Rows& R, P1Lists& lists) {
  const uint32_t i = (uint32_t)i64;
  if (act && !ts.valid(i)) {
    status[i] = kStNoTable;
    act = false;
  }
  TableView t{};
  uint32_t tid = 0, owner = i;
  Key k{0, 0};
  uint64_t v = 0, h1 = 0;
  Addr a{};
  SetProbe probe{};
  if (act) {
    tid = ts.id(i);
    t = ts.of(i);
    k = load_key(keys, i);
    v = load_val(vals, i);
    a = address_of(k, t.nb, t.seed, h1);
    probe = set_probe(ws, h1, tid, i);
  }
  const bool timers = kTimers && t.timers;
  Snap s;
  p1_fetch<kTimers>(t, a.b1, act, R, s);
  if (act) owner = set_owner(ws, ts, keys, k, tid, i, probe);
  const bool mine = act && owner == i;
  P1Bucket r{}, r2{};
  bool maybe2 = false, have2 = false;
  if (mine) {
    r = p1_bucket(a.b1, s, a.tag, timers, now, expiry);
    maybe2 = (r.bloom & a.bits) == a.bits;  // the filter allows the secondary
    have2 = maybe2 || !claimable(r.ctrl, r.dead);
  }
  p1_fetch<kTimers>(t, a.b2, have2, R, s);
  uint8_t st = 0;
  P1Work work = kP1None;
  uint32_t flip = 0;  // publication of a slot that was free: the bits of the ctrl word to flip
  int sl = -1;
  bool sticky = false;
  if (mine) {
    if (have2) r2 = p1_bucket(a.b2, s, a.tag, timers, now, expiry);
    if (!maybe2) r2.match = 0;  // not there, by the filter
    bool second;
    if ((sl = p1_search(t, r, r2, k, now, expiry, second)) >= 0) {
      st = p1_stored(t, second ? r2 : r, (uint32_t)sl, timers, work);
      if (st && second) r = r2;
    }
    if (!st) {
      for (;;) {
        uint32_t prev = 0;
        sl = claim_slot(t, r, r.b == a.b2, prev);
        if (sl >= 0) {
          work = kP1Place;
          st = kStInserted;
          sticky = kTimers && ((prev >> sl) & 1u);  // holds a dead entry
          if (!sticky) flip = claim_bit(sl) | 1u << sl | (r.b == a.b2 ? 1u << (kInsecShift + sl) : 0u);
          if (sticky && ((prev >> (kInsecShift + sl)) & 1u)) evict_displaced(t, tid, r.b, sl, ws);
          if (r.b == a.b2) {  // Sec. 4.1: displaced to the secondary
            atomicOr(reinterpret_cast<unsigned long long*>(bloom_ptr(t, a.b1)), (unsigned long long)a.bits);
            atomicAdd(moved_ptr(t, a.b1), 1u);
          }
          break;
        }
        if (sl == -2) {
          st = kStBusy;
          break;
        }
        if (r.b == a.b2) break;
        // the secondary (not read yet if the primary has filled up under the claim)
        if (!have2) {
          p1_fetch_one(t, a.b2, timers, s);
          r2 = p1_bucket(a.b2, s, a.tag, timers, now, expiry);
          r2.match = 0;
          P1Bucket none{};
          p1_search(t, r2, none, k, now, expiry, second);
        }
        r = r2;
      }
    }
    if (st) status[i] = st;
  }
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t jobs = __ballot_sync(kWarpAll, work != kP1None);
  if (work != kP1None) {
    const uint32_t j = __popc(jobs & ((1u << lane) - 1u));
    const unsigned long long bp = reinterpret_cast<unsigned long long>(bucket_ptr(t, r.b));
    const uint32_t words = (work == kP1Place ? 0x7Fu : 0x30u) | (timers ? 0x80u : 0u);
    row_chunk(R, j, 0) = make_uint4((uint32_t)k.k0, (uint32_t)(k.k0 >> 32), (uint32_t)k.k1, (uint32_t)(k.k1 >> 32));
    row_chunk(R, j, 1) = make_uint4((uint32_t)v, (uint32_t)(v >> 32), (uint32_t)bp, (uint32_t)(bp >> 32));
    row_chunk(R, j, 2) =
        make_uint4(words | (uint32_t)sl << 8 | (timers ? 0x10000u : 0u), (a.tag & 0xFFFFu) | expiry << 16, 0u, 0u);
  }
  __syncwarp();
  p1_store<kTimers>(__popc(jobs), R);
  // Entries in slots that were free are published. (A fence only where there are any: the call
  // above, which has none, 162 -> 154 us; 1M updates of a 17M-slot table 99 -> 92.)
  if (__any_sync(kWarpAll, flip != 0u)) {
    fence_acq_rel();                       // every lane's stores before any busy bit
    __syncwarp();
    if (flip) atomicXor(ctrl_ptr(t, r.b), flip);
  }
  sticky |= work == kP1Revive;
  const bool queued = mine && !st, follows = act && !mine;
  uint32_t at[3];
  lists_append<3>(lists, {ws.counters + kCntPending, ws.counters + kCntFollowers, ws.counters + kCntSticky},
                  {queued, follows, sticky}, at);
  if (queued) ws.pending[at[0]] = i;
  if (follows) write_follower(ws, at[1], i, owner);
  if (sticky) ws.sticky[at[2]] = (unsigned long long)i << 32 | r.b;
}

constexpr int kP1Threads = 128;

template <bool kTimers>
__global__ void __launch_bounds__(kP1Threads, 1024 / kP1Threads) insert_phase1(TableSet ts, const uint8_t* __restrict__ keys,
                                                             const uint64_t* __restrict__ vals, uint64_t n,
                                                             uint32_t now, uint32_t expiry,
                                                             uint8_t* __restrict__ status, Workspace ws) {
  __shared__ P1Rows rows[kP1Threads / 32];
  __shared__ P1Lists lists;
  lists_init(lists);
  pdl_wait();
  const uint64_t i = blockIdx.x * (uint64_t)kP1Threads + threadIdx.x;
  phase1_one<kTimers>(ts, keys, vals, now, expiry, status, ws, i, i < n, rows[threadIdx.x >> 5], lists);
}

// --------------------------------------------------------------- phase 2
// Search budgets of the displacement passes after move1 (queue in shared
// memory, at most 48 KB per block): the grid pass searches 96 buckets up to 4
// moves deep, one thread per key (many keys, so the searches in flight matter
// most; a list of at most kGridWarpKeys keys runs one warp per key); the
// second pass 192 buckets, 5 moves, and the last pass 2048 buckets, 6 moves,
// one warp per key (few keys, so the time of one search matters most; the
// sequential CPU reference searches 1024 buckets, 5 moves). Each
// later pass takes on at most kSecondPassKeys / kLastPassKeys keys, which
// bounds the time a batch spends on a table that is full: the rest are FULL
// without a search. Near LF 0.98 the second pass still places about two
// thirds of the keys it searches, so its share is wide.
//
// Within one insert call no bucket gains a free or dead slot: phase 1 fills
// them, a path ends by filling one, every move along it vacates a slot that
// the next move (or the key) refills, and `now` is fixed. A key queued by
// phase 1 found both its buckets without a free or dead slot, so the passes
// search from them without re-checking the roots.
constexpr int kP2Threads = 64;
constexpr uint32_t kSecondPassKeys = 65536;  // keys the second pass takes on
constexpr uint32_t kLastPassKeys = 1024;     // keys the last pass takes on
// A grid search list this short runs one warp per key: the slowest search sets
// the pass's time, and a warp takes a level of a search in two round trips.
constexpr uint32_t kGridWarpKeys = 1024;
constexpr int kMaxDepth = 6;
constexpr int kPathBuckets = kMaxDepth + 1;
constexpr int kMaxLocks = kPathBuckets + 1;   // the path plus the key's primary

struct Node {
  uint32_t bucket;
  int16_t parent;
  uint8_t slot;   // slot of the parent bucket whose entry moves into this bucket
  uint8_t depth;
};

// One thread's search queue inside a block's shared array stored node-major
// (node j of every thread side by side), so that the threads of a warp touch
// consecutive words and never the same bank.
struct Queue {
  Node* base;
  int stride;
  __device__ __forceinline__ Node& operator[](int i) const { return base[i * stride]; }
};

// Breadth-first search over buckets from b1 and b2 by one thread (lock-free
// reads; the path is re-validated under its locks). Expanding a bucket issues
// the reads of its control word and the keys of its 8 slots together (each
// entry's other bucket takes one hash, chosen by its in_secondary bit), then
// the control-word (and expiry) reads of the 8 buckets those entries can move
// to, so one level of the search costs two memory round trips; a child with a
// free or dead slot ends the search (the first such child in queue order, i.e.
// a shortest path). A child is not queued if it is one of the roots, a bucket
// on its parent's path or an earlier sibling, so no path holds a bucket twice;
// a bucket reached again by another branch takes a second queue node (a scan
// of the whole queue for it cost more than the node: most repeats are an
// entry's way back to the bucket it came from, which the path test catches).
// Returns the node index of the bucket with the hole (in hole), or -1.
template <int kBfsNodes, int kBfsDepth>
__device__ int bfs(const TableView& t, const Addr& a, uint32_t now, const Queue& q, uint32_t& hole) {
  static_assert(kBfsNodes < 32768, "parent index exceeds its field");
  int nq = 0;
  q[nq++] = Node{a.b1, -1, 0, 0};
  q[nq++] = Node{a.b2, -1, 0, 0};
  // A hole is only ever found on a newly queued bucket, so the search ends
  // when the queue is full.
  for (int qi = 0; qi < nq && nq < kBfsNodes; ++qi) {
    const Node cur = q[qi];
    if (cur.depth >= kBfsDepth) continue;
    uint64_t k0[kSlots], k1[kSlots];
    const uint32_t cc = load_bucket_keys(t, cur.bucket, k0, k1);
    uint32_t y[kSlots], cy[kSlots];
    uint64_t e0[kSlots], e1[kSlots];
#pragma unroll
    for (uint32_t sl = 0; sl < kSlots; ++sl)
      y[sl] = other_bucket(Key{k0[sl], k1[sl]}, cur.bucket, (cc >> (kInsecShift + sl)) & 1u, t.nb, t.seed);
#pragma unroll
    for (uint32_t sl = 0; sl < kSlots; ++sl) {
      cy[sl] = ld32_cg(ctrl_ptr(t, y[sl]));
      if (t.timers) {
        ld128_cg(expiry_ptr(t, y[sl], 0), e0[sl], e1[sl]);
      } else {
        e0[sl] = e1[sl] = 0;
      }
    }
    // children to skip: a root, a bucket on cur's path (cur and its ancestors), an earlier sibling
    uint32_t path_b[kBfsDepth + 1];
    int node = qi;
#pragma unroll
    for (int d = 0; d <= kBfsDepth; ++d) {
      path_b[d] = node >= 0 ? q[node].bucket : a.b1;  // past the root: a root again, already tested
      node = node >= 0 ? q[node].parent : -1;
    }
    uint32_t skip = 0;
#pragma unroll
    for (uint32_t sl = 0; sl < kSlots; ++sl) {
      bool hit = y[sl] == a.b1 || y[sl] == a.b2;
#pragma unroll
      for (int d = 0; d <= kBfsDepth; ++d) hit |= path_b[d] == y[sl];
#pragma unroll
      for (uint32_t o = 0; o < sl; ++o) hit |= y[o] == y[sl];
      skip |= (uint32_t)hit << sl;
    }
    for (uint32_t sl = 0; sl < kSlots && nq < kBfsNodes; ++sl) {
      if ((skip >> sl) & 1u) continue;
      q[nq] = Node{y[sl], (int16_t)qi, (uint8_t)sl, (uint8_t)(cur.depth + 1)};
      Snap s;
      s.e0 = e0[sl];
      s.e1 = e1[sl];
      const uint32_t f = free_mask(t, cy[sl], s, now);
      ++nq;
      if (f) {
        hole = __ffs(f) - 1;
        return nq - 1;
      }
    }
  }
  return -1;
}

// The same search run by a whole warp for one key. A round expands up to 32
// queued buckets at once, one per lane, with the thread form's two round trips
// (a lane's bucket keys and control word, then the control words of the 8
// buckets its entries can move to), so a level of the search costs two round
// trips however wide it is. The children of a round enter the queue in queue
// order (lane, then slot; the queue stays sorted by depth), each bucket once:
// the visited set is a shared open-addressing table updated with atomicCAS,
// sized for the queue plus one round of children. The hole is the first child
// in queue order with a free or dead slot, a shortest path as in the thread
// form. q: the warp's queue (kBfsNodes nodes); seen: its set. Every lane
// returns the same node index (or -1) and hole.
template <int kBfsNodes>
struct WarpSeen {
  // smallest power of two at least 1.5 x (kBfsNodes + the 256 children of a round)
  static constexpr uint32_t kNeed = (kBfsNodes + 256) * 3 / 2;
  static constexpr uint32_t kSize = kNeed <= 1024 ? 1024 : (kNeed <= 2048 ? 2048 : (kNeed <= 4096 ? 4096 : 8192));
  static_assert(kNeed <= 8192, "visited set too large");
};

template <uint32_t kSize>
__device__ __forceinline__ bool seen_insert_shared(uint32_t* seen, uint32_t b) {
  uint32_t h = (b * 0x9E3779B1u) & (kSize - 1);
  for (uint32_t probe = 0; probe < kSize; ++probe) {
    const uint32_t old = atomicCAS(&seen[h], 0xFFFFFFFFu, b);
    if (old == 0xFFFFFFFFu) return true;
    if (old == b) return false;
    h = (h + 1) & (kSize - 1);
  }
  return false;  // not reached: the set is sized for every bucket a search can meet
}

template <int kBfsNodes, int kBfsDepth>
__device__ int bfs_warp(const TableView& t, const Addr& a, uint32_t now, Node* q, uint32_t* seen, uint32_t& hole) {
  constexpr uint32_t kSeen = WarpSeen<kBfsNodes>::kSize;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t j = lane; j < kSeen; j += 32) seen[j] = 0xFFFFFFFFu;
  __syncwarp();
  if (lane == 0) {
    q[0] = Node{a.b1, -1, 0, 0};
    q[1] = Node{a.b2, -1, 0, 0};
    seen_insert_shared<kSeen>(seen, a.b1);
    seen_insert_shared<kSeen>(seen, a.b2);
  }
  __syncwarp();
  int nq = 2;
  for (int head = 0; head < nq && nq < kBfsNodes;) {
    const int chunk_end = min(nq, head + 32);
    const int qi = head + (int)lane;
    Node cur{0, -1, 0, (uint8_t)kBfsDepth};
    if (qi < chunk_end) cur = q[qi];
    uint32_t y[kSlots];
    uint32_t fresh = 0;   // children this lane queues
    uint64_t holes = 0;   // their free or dead slots, 8 bits per child
    if (cur.depth < kBfsDepth) {
      uint64_t k0[kSlots], k1[kSlots];
      const uint32_t cc = load_bucket_keys(t, cur.bucket, k0, k1);
      uint32_t cy[kSlots];
      uint64_t e0[kSlots], e1[kSlots];
#pragma unroll
      for (uint32_t sl = 0; sl < kSlots; ++sl)
        y[sl] = other_bucket(Key{k0[sl], k1[sl]}, cur.bucket, (cc >> (kInsecShift + sl)) & 1u, t.nb, t.seed);
#pragma unroll
      for (uint32_t sl = 0; sl < kSlots; ++sl) {
        cy[sl] = ld32_cg(ctrl_ptr(t, y[sl]));
        if (t.timers) {
          ld128_cg(expiry_ptr(t, y[sl], 0), e0[sl], e1[sl]);
        } else {
          e0[sl] = e1[sl] = 0;
        }
      }
#pragma unroll
      for (uint32_t sl = 0; sl < kSlots; ++sl) {
        if (!seen_insert_shared<kSeen>(seen, y[sl])) continue;
        fresh |= 1u << sl;
        Snap s;
        s.e0 = e0[sl];
        s.e1 = e1[sl];
        holes |= (uint64_t)free_mask(t, cy[sl], s, now) << (8 * sl);
      }
    }
    // queue positions: the children of lower lanes first
    const uint32_t cnt = __popc(fresh);
    uint32_t incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(kWarpAll, incl, d);
      if ((int)lane >= d) incl += o;
    }
    const uint32_t total = __shfl_sync(kWarpAll, incl, 31);
    int pos = nq + (int)(incl - cnt);
    int best = 0x7FFFFFFF;  // this lane's first queued child with room
    uint32_t best_hole = 0;
#pragma unroll
    for (uint32_t sl = 0; sl < kSlots; ++sl) {
      if (!((fresh >> sl) & 1u)) continue;
      if (pos < kBfsNodes) {
        q[pos] = Node{y[sl], (int16_t)qi, (uint8_t)sl, (uint8_t)(cur.depth + 1)};
        const uint32_t f = (uint32_t)(holes >> (8 * sl)) & 0xFFu;
        if (f && best == 0x7FFFFFFF) {
          best = pos;
          best_hole = __ffs(f) - 1;
        }
      }
      ++pos;
    }
    __syncwarp();  // the new nodes before any lane reads them
    const int wbest = __reduce_min_sync(kWarpAll, best);
    if (wbest != 0x7FFFFFFF) {
      const uint32_t src = __ffs(__ballot_sync(kWarpAll, best == wbest)) - 1;
      hole = __shfl_sync(kWarpAll, best_hole, src);
      return wbest;
    }
    nq = min(nq + (int)total, kBfsNodes);
    head = chunk_end;
  }
  return -1;
}

// Move the entry in slot sx of locked bucket x to the free slot sy of locked
// bucket y, its other bucket. Sec. 4.1: a move from the primary to the
// secondary sets the entry's bits in the primary's filter and increments its
// counter; the reverse move decrements the counter and resets the filter at
// zero (safe: filter bits of y are only ever set under y's lock, held here).
__device__ void move_locked(const TableView& t, uint32_t x, uint32_t sx, uint32_t& cx, uint32_t y, uint32_t sy,
                            uint32_t& cy) {
  uint64_t k0, k1;
  ld128_cg(key_ptr(t, x, sx), k0, k1);
  const uint64_t v = ld64_cg(value_ptr(t, x, sx));
  const Addr e = address_of(Key{k0, k1}, t.nb, t.seed);
  st128_cg(key_ptr(t, y, sy), k0, k1);
  st64_cg(value_ptr(t, y, sy), v);
  st16_cg(tag_ptr(t, y, sy), e.tag);
  if (t.timers) st16_cg(expiry_ptr(t, y, sy), ld16_cg(expiry_ptr(t, x, sx)));
  cy |= 1u << sy;
  if (e.b1 == x) {
    cy |= 1u << (kInsecShift + sy);
    atomicOr(reinterpret_cast<unsigned long long*>(bloom_ptr(t, x)), (unsigned long long)e.bits);
    atomicAdd(moved_ptr(t, x), 1u);
  } else {
    cy &= ~(1u << (kInsecShift + sy));
    if (atomicSub(moved_ptr(t, y), 1u) == 1u) atomicExch(reinterpret_cast<unsigned long long*>(bloom_ptr(t, y)), 0ull);
  }
  cx &= ~((1u << sx) | (1u << (kInsecShift + sx)));
}

// Execute a cuckoo path atomically: lock every bucket on it plus the key's
// primary (in index order), check that each entry still sits where the search
// saw it and still has the next bucket as its other bucket and that the end
// slot is still free or dead, then move the entries backwards (each into the
// hole ahead of it) and store the new key in the hole left in the root bucket.
// path[0] is the root (b1 or b2), path[len] the bucket with the hole; slot[j]
// is the slot of path[j] whose entry moves to path[j + 1].
// 1 placed, 0 stale path, -1 lock timeout.
__device__ int execute_path(const TableView& t, uint32_t tid, const uint32_t (&path)[kPathBuckets],
                            const uint32_t (&slot)[kPathBuckets], int len, uint32_t hole, const Key& k, uint64_t v,
                            const Addr& a, uint32_t now, uint32_t expiry, const Workspace& ws) {
  uint32_t lk[kMaxLocks], cw[kMaxLocks];
  int nl = 0;
  bool has_b1 = false;
  for (int j = 0; j <= len; ++j) {
    lk[nl++] = path[j];
    has_b1 |= (path[j] == a.b1);
  }
  if (!has_b1) lk[nl++] = a.b1;
  for (int i = 1; i < nl; ++i)  // insertion sort: a global lock order
    for (int j = i; j > 0 && lk[j - 1] > lk[j]; --j) {
      const uint32_t tmp = lk[j];
      lk[j] = lk[j - 1];
      lk[j - 1] = tmp;
    }
  for (int i = 0; i < nl; ++i) {
    if (!lock_bucket(t, lk[i], cw[i])) {
      for (int j = i - 1; j >= 0; --j) unlock_bucket(t, lk[j], cw[j]);
      return -1;
    }
  }
  auto idx = [&](uint32_t b) {
    int r = 0;
    for (int i = 0; i < nl; ++i) r = (lk[i] == b) ? i : r;
    return r;
  };
  bool ok = true;
  for (int j = 0; j < len && ok; ++j) {
    if (!((cw[idx(path[j])] >> slot[j]) & 1u)) {
      ok = false;
      break;
    }
    Key ek;
    ld128_cg(key_ptr(t, path[j], slot[j]), ek.k0, ek.k1);
    const Addr e = address_of(ek, t.nb, t.seed);
    const uint32_t other = (e.b1 == path[j]) ? e.b2 : (e.b2 == path[j] ? e.b1 : 0xFFFFFFFFu);
    ok = (other == path[j + 1]);
  }
  const int ie = idx(path[len]);
  const bool end_busy = (cw[ie] >> hole) & 1u;
  if (ok && end_busy) ok = t.timers && !alive16(ld16_cg(expiry_ptr(t, path[len], hole)), now);
  int rc = 0;
  if (ok) {
    if (end_busy) evict_entry(t, tid, path[len], hole, cw[ie], ws);
    uint32_t dst_s = hole;
    for (int j = len - 1; j >= 0; --j) {
      move_locked(t, path[j], slot[j], cw[idx(path[j])], path[j + 1], dst_s, cw[idx(path[j + 1])]);
      dst_s = slot[j];
    }
    place_entry(t, path[0], dst_s, k, v, a, expiry, cw[idx(path[0])]);
    rc = 1;
  }
  for (int i = nl - 1; i >= 0; --i) unlock_bucket(t, lk[i], cw[i]);
  return rc;
}

// The same by a whole warp, for the path that ends at node `end` of its queue q
// (hole: the slot there): lane j holds path[j] (and slot[j] of the entry that
// leaves it), lane len + 1 the key's primary if it is not the root. The locks
// are taken, the entries read, checked and written, and the locks released by
// all lanes at once, so that a path of any length takes the round trips of one
// move (one thread took two or three per bucket; inserts of 8K and 32K new keys
// into 1M slots at load 0.85: 65 -> 61 and 81 -> 75 us). Every lane returns the
// result.
__device__ int execute_path_warp(const TableView& t, uint32_t tid, const Node* q, int end, uint32_t hole, const Key& k,
                                 uint64_t v, const Addr& a, uint32_t now, uint32_t expiry, const Workspace& ws) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t len = q[end].depth;
  uint32_t b = 0, s = hole;  // this lane's bucket and the slot that it fills (and, before the end, empties first)
  uint32_t root = 0;
  for (int node = end; node >= 0;) {
    const Node nd = q[node];
    if (nd.depth == lane) b = nd.bucket;
    if (nd.depth == lane + 1u) s = nd.slot;
    if (nd.depth == 0) root = nd.bucket;
    node = nd.parent;
  }
  const bool on_path = lane <= len, moves = lane < len;
  const bool is_b1 = lane == len + 1u && root != a.b1;
  if (is_b1) b = a.b1;
  const bool act = on_path || is_b1;
  // locks: all bits at once, else one by one in index order (as lock_buckets)
  uint32_t cw = 0;
  if (act) cw = or_relaxed(ctrl_ptr(t, b), kLockBit);
  if (__any_sync(kWarpAll, act && (cw & kLockBit))) {
    if (act && !(cw & kLockBit)) and_relaxed(ctrl_ptr(t, b), ~kLockBit);  // nothing written: drop it
    const uint32_t n = __popc(__ballot_sync(kWarpAll, act));
    uint32_t rank = 0;
    for (uint32_t j = 0; j < n; ++j) rank += __shfl_sync(kWarpAll, b, j) < b;  // lanes 0..n-1 are the active ones
    bool locked = false;
    for (uint32_t r = 0; r < n; ++r) {
      bool gave_up = false;
      if (act && rank == r) {
        locked = lock_bucket(t, b, cw);
        gave_up = !locked;
      }
      if (__any_sync(kWarpAll, gave_up)) {
        if (locked) unlock_bucket(t, b, cw);
        return -1;
      }
    }
  }
  fence_acq_rel();
  // the entries that move
  Key e{0, 0};
  uint64_t ev = 0;
  uint32_t exp = 0;
  if (moves) {
    ld128_cg(key_ptr(t, b, s), e.k0, e.k1);
    ev = ld64_cg(value_ptr(t, b, s));
  }
  if (on_path && t.timers) exp = ld16_cg(expiry_ptr(t, b, s));
  const bool insec = (cw >> (kInsecShift + s)) & 1u, busy = (cw >> s) & 1u;
  const uint64_t h1 = hash_key(e, t.seed), h2 = hash_key(e, t.seed ^ kSeed2Xor);
  const uint32_t b2 = reduce(h2, t.nb);
  const uint32_t other = insec ? reduce(h1, t.nb) : (b2 != b ? b2 : (b + 1 == (uint32_t)t.nb ? 0u : b + 1));
  const uint32_t next_b = __shfl_down_sync(kWarpAll, b, 1), next_s = __shfl_down_sync(kWarpAll, s, 1);
  const bool came_insec = __shfl_up_sync(kWarpAll, (int)insec, 1);  // the entry that comes here was in its secondary
  bool ok = true;
  if (moves) ok = busy && other == next_b;
  if (lane == len) ok = !busy || (t.timers && !alive16(exp, now));
  ok = __all_sync(kWarpAll, ok);
  const uint32_t old_cw = cw;
  if (ok && lane == len && busy && insec) evict_displaced(t, tid, b, s, ws);  // reads the dead entry's key
  __syncwarp();
  if (ok) {
    if (moves) {
      st128_cg(key_ptr(t, next_b, next_s), e.k0, e.k1);
      st64_cg(value_ptr(t, next_b, next_s), ev);
      st16_cg(tag_ptr(t, next_b, next_s), (uint32_t)(h1 & 0xFFFF));
      if (t.timers) st16_cg(expiry_ptr(t, next_b, next_s), exp);
    }
    // Sec. 4.1 on this lane's bucket: an entry that leaves it for its secondary adds its bits and
    // one to the counter, one that comes home to it takes one off, at zero with the filter
    const bool leaves = moves && !insec, home = on_path && lane > 0 && came_insec;
    if (leaves || is_b1) {
      const uint64_t bits = is_b1 ? a.bits : (1ull << (h2 & 63)) | (1ull << ((h2 >> 6) & 63));
      atomicOr(reinterpret_cast<unsigned long long*>(bloom_ptr(t, b)), (unsigned long long)bits);
      if (!home) atomicAdd(moved_ptr(t, b), 1u);
    } else if (home && atomicSub(moved_ptr(t, b), 1u) == 1u) {
      atomicExch(reinterpret_cast<unsigned long long*>(bloom_ptr(t, b)), 0ull);
    }
    if (lane == 0) {  // the new key, into the slot that the root's entry leaves
      st128_cg(key_ptr(t, b, s), k.k0, k.k1);
      st64_cg(value_ptr(t, b, s), v);
      st16_cg(tag_ptr(t, b, s), a.tag);
      if (t.timers) st16_cg(expiry_ptr(t, b, s), expiry);
    }
    if (on_path) {
      const bool now_insec = lane == 0 ? b == a.b2 : !came_insec;
      cw = (cw & ~(1u << (kInsecShift + s))) | 1u << s | (now_insec ? 1u << (kInsecShift + s) : 0u);
    }
  }
  fence_acq_rel();
  __syncwarp();
  if (act) exch_relaxed(ctrl_ptr(t, b), (ok ? cw : old_cw) & ~kLockBit);
  return ok ? 1 : 0;
}

// A cuckoo path of length one, found by the one-move pass: the entry in slot
// sx of root x (a root of key k: a.b1 or a.b2) moves to free (or dead) slot
// hole of its other bucket y, and k takes slot sx. Under the locks of x, y and
// (when x is k's secondary) k's primary, the path is valid if slot sx is busy
// and its entry's other bucket, from the key and in_secondary bit read under
// the locks, is still y, and y still has room: the hole if it is still free or
// dead, else any slot of y that is free now. The entry's value
// and expiry are read in the same round trip as its key; its tag and filter
// bits come from its two hashes. The moves are those of execute_path. 1
// placed, 0 stale path, -1 lock timeout.
__device__ int execute_move1(const TableView& t, uint32_t tid, uint32_t x, uint32_t sx, uint32_t y, uint32_t hole,
                             const Key& k, uint64_t v, const Addr& a, uint32_t now, uint32_t expiry,
                             const Workspace& ws) {
  uint32_t lk[3], cw[3];
  int nl = 0;
  // x and y are distinct and differ from a.b1 unless x == a.b1 (the search skips y in {b1, b2})
  const uint32_t u0 = x < y ? x : y, u1 = x < y ? y : x;
  if (x == a.b1) {
    lk[0] = u0;
    lk[1] = u1;
    nl = 2;
  } else {
    const uint32_t p = a.b1;
    lk[0] = p < u0 ? p : u0;
    lk[1] = p < u0 ? u0 : (p < u1 ? p : u1);
    lk[2] = p < u1 ? u1 : p;
    nl = 3;
  }
  if (!lock_buckets<3>(t, lk, nl, cw)) return -1;
  int ix = 0, iy = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i < nl && lk[i] == x) ix = i;
    if (i < nl && lk[i] == y) iy = i;
  }
  Key ek;
  ld128_cg(key_ptr(t, x, sx), ek.k0, ek.k1);
  const uint64_t ev = ld64_cg(value_ptr(t, x, sx));
  const uint32_t eexp = t.timers ? ld16_cg(expiry_ptr(t, x, sx)) : 0u;
  const uint32_t hexp = t.timers ? ld16_cg(expiry_ptr(t, y, hole)) : 0u;
  const bool insec = (cw[ix] >> (kInsecShift + sx)) & 1u;
  // H1 gives the entry's tag and the primary of an entry in its secondary, H2 the secondary
  // (and filter bits) of an entry in its primary; hashing beats a fourth memory request
  const uint64_t h1 = hash_key(ek, t.seed), h2 = hash_key(ek, t.seed ^ kSeed2Xor);
  const uint32_t b2 = reduce(h2, t.nb);
  const uint32_t other = insec ? reduce(h1, t.nb) : (b2 != x ? b2 : (x + 1 == (uint32_t)t.nb ? 0u : x + 1));
  const uint32_t etag = (uint32_t)(h1 & 0xFFFF);
  const uint64_t bits = (1ull << (h2 & 63)) | (1ull << ((h2 >> 6) & 63));
  bool ok = ((cw[ix] >> sx) & 1u) && other == y;
  bool end_busy = (cw[iy] >> hole) & 1u;
  if (end_busy && !(t.timers && !alive16(hexp, now))) {
    // another key took the hole since the search: any slot of y that is free now will do
    const uint32_t fr = ~cw[iy] & kBusyMask;
    if (fr) {
      hole = __ffs(fr) - 1;
      end_busy = false;
    }
  }
  if (ok && end_busy) ok = t.timers && !alive16(hexp, now);
  if (ok) {
    if (end_busy) evict_entry(t, tid, y, hole, cw[iy], ws);
    st128_cg(key_ptr(t, y, hole), ek.k0, ek.k1);
    st64_cg(value_ptr(t, y, hole), ev);
    st16_cg(tag_ptr(t, y, hole), etag);
    if (t.timers) st16_cg(expiry_ptr(t, y, hole), eexp);
    cw[iy] |= 1u << hole;
    if (!insec) {  // Sec. 4.1: primary x -> secondary y: x's filter gets the entry's bits, its counter + 1
      cw[iy] |= 1u << (kInsecShift + hole);
      atomicOr(reinterpret_cast<unsigned long long*>(bloom_ptr(t, x)), (unsigned long long)bits);
      atomicAdd(moved_ptr(t, x), 1u);
    } else {  // secondary x -> primary y: y's counter - 1, its filter reset at zero (y is locked)
      cw[iy] &= ~(1u << (kInsecShift + hole));
      if (atomicSub(moved_ptr(t, y), 1u) == 1u) atomicExch(reinterpret_cast<unsigned long long*>(bloom_ptr(t, y)), 0ull);
    }
    cw[ix] &= ~((1u << sx) | (1u << (kInsecShift + sx)));
    place_entry(t, x, sx, k, v, a, expiry, cw[ix]);
  }
  unlock_buckets<3>(t, lk, nl, cw);
  return ok ? 1 : 0;
}

// One-move pass over list[0..count): for each key, the entries
// of b1 and then of b2 are read with the buckets they can move to (two memory
// round trips per root: the root's keys and control word, then the control
// words of the buckets its entries can move to; each entry's other bucket
// takes one hash, chosen by its in_secondary bit); the first entry whose other
// bucket has a free or dead slot gives a cuckoo path of length one, executed
// under locks (execute_move1). Keys without one, or whose path went stale, are
// appended to `next`. The key's value is requested before the search.
// worker / workers: this thread's index among the threads sharing the pass.
__device__ void move1_range(const TableSet& ts, const uint8_t* __restrict__ keys, const uint64_t* __restrict__ vals,
                            uint32_t now, uint32_t expiry, uint8_t* __restrict__ status, const Workspace& ws,
                            const uint32_t* list, uint32_t count, uint32_t* next, uint32_t* next_count,
                            uint32_t worker, uint32_t workers) {
  for (uint32_t j = worker; j < count; j += workers) {
    const uint32_t i = list[j];
    const TableView t = ts.of(i);
    const uint64_t v = load_val(vals, i);
    const Key k = load_key(keys, i);
    const Addr a = address_of(k, t.nb, t.seed);
    uint32_t x = 0, sx = 0, y = 0, hole = 0;
    bool found = false;
    for (int r = 0; r < 2 && !found; ++r) {
      const uint32_t root = r ? a.b2 : a.b1;
      uint64_t k0[kSlots], k1[kSlots];
      const uint32_t cr = load_bucket_keys(t, root, k0, k1);
      uint32_t yy[kSlots];
#pragma unroll
      for (uint32_t sl = 0; sl < kSlots; ++sl)
        yy[sl] = other_bucket(Key{k0[sl], k1[sl]}, root, (cr >> (kInsecShift + sl)) & 1u, t.nb, t.seed);
      // the buckets the entries can move to, kMoveGroup at a time: most keys find room among the
      // first ones, and each bucket read is a memory request of its own
      for (uint32_t g = 0; g < kSlots && !found; g += kMoveGroup) {
        uint32_t cy[kMoveGroup];
        uint64_t e0[kMoveGroup], e1[kMoveGroup];
#pragma unroll
        for (uint32_t q = 0; q < kMoveGroup; ++q) {
          cy[q] = ld32_cg(ctrl_ptr(t, yy[g + q]));
          if (t.timers) {
            ld128_cg(expiry_ptr(t, yy[g + q], 0), e0[q], e1[q]);
          } else {
            e0[q] = e1[q] = 0;
          }
        }
#pragma unroll
        for (uint32_t q = 0; q < kMoveGroup; ++q) {
          const uint32_t sl = g + q;
          if (found || yy[sl] == a.b1 || yy[sl] == a.b2) continue;  // the roots have no room
          Snap s;
          s.e0 = e0[q];
          s.e1 = e1[q];
          const uint32_t f = free_mask(t, cy[q], s, now);
          if (f) {
            x = root;
            sx = sl;
            y = yy[sl];
            hole = __ffs(f) - 1;
            found = true;
          }
        }
      }
    }
    int rc = 0;
    if (found) rc = execute_move1(t, ts.id(i), x, sx, y, hole, k, v, a, now, expiry, ws);
    if (rc == 0) {
      next[atomicAdd(next_count, 1u)] = i;
    } else {
      if (rc < 0) latch_error(t, kErrLockTimeout);
      status[i] = rc > 0 ? kStInserted : kStBusy;
    }
  }
}

// The same pass with half a warp per key, for a list so short that the time of
// one key sets the pass's: lane r * 8 + sl of the half reads slot sl of root r,
// so that both roots' keys come in one round trip and all 16 buckets their
// entries can move to in a second, where a thread takes up to ten. The first
// one with room, in the thread form's order, is the path; its lane executes it.
// half / halves: this half warp's index among those sharing the pass (whole
// warps call this).
__device__ void move1_range_half(const TableSet& ts, const uint8_t* __restrict__ keys,
                                 const uint64_t* __restrict__ vals, uint32_t now, uint32_t expiry,
                                 uint8_t* __restrict__ status, const Workspace& ws, const uint32_t* list,
                                 uint32_t count, uint32_t* next, uint32_t* next_count, uint32_t half,
                                 uint32_t halves) {
  const uint32_t lane = threadIdx.x & 15u, sl = lane & 7u;
  const uint32_t shift = threadIdx.x & 16u;  // of this half's lanes in a ballot
  for (uint32_t first = half & ~1u; first < count; first += halves) {  // the same for both halves
    const uint32_t j = first + (half & 1u);
    const bool act = j < count;
    const uint32_t i = act ? list[j] : 0u;
    TableView t{};
    Key k{0, 0};
    uint64_t v = 0;
    Addr a{};
    uint32_t x = 0, y = 0, f = 0;
    if (act) {
      t = ts.of(i);
      v = load_val(vals, i);
      k = load_key(keys, i);
      a = address_of(k, t.nb, t.seed);
      x = lane < 8u ? a.b1 : a.b2;
      const uint32_t cr = ld32_cg(ctrl_ptr(t, x));
      Key e;
      ld128_cg(key_ptr(t, x, sl), e.k0, e.k1);
      y = other_bucket(e, x, (cr >> (kInsecShift + sl)) & 1u, t.nb, t.seed);
      Snap s;
      const uint32_t cy = ld32_cg(ctrl_ptr(t, y));
      s.e0 = s.e1 = 0;
      if (t.timers) ld128_cg(expiry_ptr(t, y, 0), s.e0, s.e1);
      if (y != a.b1 && y != a.b2) f = free_mask(t, cy, s, now);  // the roots have no room
    }
    const uint32_t with_room = (__ballot_sync(kWarpAll, f != 0u) >> shift) & 0xFFFFu;
    if (act && (with_room ? lane == (uint32_t)__ffs(with_room) - 1u : lane == 0u)) {
      int rc = 0;
      if (with_room) rc = execute_move1(t, ts.id(i), x, sl, y, __ffs(f) - 1, k, v, a, now, expiry, ws);
      if (rc == 0) {
        next[atomicAdd(next_count, 1u)] = i;
      } else {
        if (rc < 0) latch_error(t, kErrLockTimeout);
        status[i] = rc > 0 ? kStInserted : kStBusy;
      }
    }
    __syncwarp();
  }
}

// The longest list that runs half a warp per key (if there are as many halves):
// a list of 4.9K keys of a 134M-slot table 28 -> 19 us, of 7K keys with timers 22
// -> 20 us; 13K keys 82 -> 84 us of a whole call, 55K keys 115 -> 147 us.
constexpr uint32_t kMoveHalfKeys = 8192;

__global__ void __launch_bounds__(kThreads, 1) insert_move1(TableSet ts, const uint8_t* __restrict__ keys,
                                                         const uint64_t* __restrict__ vals, uint32_t now,
                                                         uint32_t expiry, uint8_t* __restrict__ status, Workspace ws,
                                                         const uint32_t* list, const uint32_t* count_ptr,
                                                         uint32_t* next, uint32_t* next_count) {
  pdl_wait();
  const uint32_t worker = blockIdx.x * blockDim.x + threadIdx.x, workers = gridDim.x * blockDim.x;
  const uint32_t count = ld32_cg(count_ptr);
  if (count <= min(kMoveHalfKeys, workers / 16u)) {
    move1_range_half(ts, keys, vals, now, expiry, status, ws, list, count, next, next_count, worker / 16u,
                     workers / 16u);
  } else {
    move1_range(ts, keys, vals, now, expiry, status, ws, list, count, next, next_count, worker, workers);
  }
}

// Displacement pass over `list` (count in *count). Keys that find no path
// are appended to `retry` (when given) for a second, low-contention pass;
// otherwise they are FULL. q: this thread's search queue.
template <int kBfsNodes, int kBfsDepth>
__device__ void phase2_range(const TableSet& ts, const uint8_t* __restrict__ keys, const uint64_t* __restrict__ vals,
                             uint32_t now, uint32_t expiry, uint8_t* __restrict__ status, const Workspace& ws,
                             const uint32_t* list, uint32_t listed, uint32_t* retry, uint32_t* retry_count,
                             uint32_t max_keys, const Queue& q, uint32_t worker, uint32_t workers) {
  static_assert(kBfsDepth <= kMaxDepth, "path longer than the lock set");
  const uint32_t count = min(listed, max_keys);
  // A later pass searches wider but alone; when many keys reach it the table
  // is full rather than contended, and those beyond max_keys are FULL at once.
  for (uint32_t j = count + worker; j < listed; j += workers) status[list[j]] = kStFull;
  for (uint32_t j = worker; j < count; j += workers) {
    const uint32_t i = list[j];
    const TableView t = ts.of(i);
    const uint32_t tid = ts.id(i);
    const uint64_t v = load_val(vals, i);
    const Key k = load_key(keys, i);
    const Addr a = address_of(k, t.nb, t.seed);
    uint8_t st = kStFull;
    for (int attempt = 0; attempt < kPathAttempts; ++attempt) {
      uint32_t hole = 0;
      const int end = bfs<kBfsNodes, kBfsDepth>(t, a, now, q, hole);
      if (end < 0) break;  // no cuckoo path within the search bound: FULL
      uint32_t path[kPathBuckets], slot[kPathBuckets];
      const int len = q[end].depth;
      for (int node = end; node >= 0; node = q[node].parent) {
        path[q[node].depth] = q[node].bucket;
        if (q[node].depth > 0) slot[q[node].depth - 1] = q[node].slot;
      }
      const int r = execute_path(t, tid, path, slot, len, hole, k, v, a, now, expiry, ws);
      if (r != 0) {
        st = r > 0 ? kStInserted : kStBusy;
        break;
      }
    }
    if (st == kStFull && retry) {
      retry[atomicAdd(retry_count, 1u)] = i;
      continue;
    }
    if (st == kStBusy) latch_error(t, kErrLockTimeout);
    status[i] = st;
  }
}

// One key's search by a whole warp (bfs_warp) and the execution of the path it
// finds: INSERTED, BUSY, or FULL if there is no path within the search's bounds.
template <int kBfsNodes, int kBfsDepth>
__device__ uint8_t search_warp(const TableView& t, uint32_t tid, const Key& k, uint64_t v, const Addr& a, uint32_t now,
                               uint32_t expiry, const Workspace& ws, Node* q, uint32_t* seen) {
  static_assert(kBfsDepth <= kMaxDepth, "path longer than the lock set");
  for (int attempt = 0; attempt < kPathAttempts; ++attempt) {
    uint32_t hole = 0;
    const int end = bfs_warp<kBfsNodes, kBfsDepth>(t, a, now, q, seen, hole);
    if (end < 0) break;
    const int r = execute_path_warp(t, tid, q, end, hole, k, v, a, now, expiry, ws);
    __syncwarp();  // every lane is done with the queue
    if (r != 0) return r > 0 ? kStInserted : kStBusy;
  }
  return kStFull;
}

// phase2_range with one warp per key (bfs_warp): warp / warps are this warp's
// index among the warps sharing the pass; q and seen are the warp's own.
// listed: the list's length (read by the caller after the list was final).
template <int kBfsNodes, int kBfsDepth>
__device__ void phase2_range_warp(const TableSet& ts, const uint8_t* __restrict__ keys,
                                  const uint64_t* __restrict__ vals, uint32_t now, uint32_t expiry,
                                  uint8_t* __restrict__ status, const Workspace& ws, const uint32_t* list,
                                  uint32_t listed, uint32_t* retry, uint32_t* retry_count,
                                  uint32_t max_keys, Node* q, uint32_t* seen, uint32_t warp, uint32_t warps) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t count = min(listed, max_keys);
  for (uint32_t j = count + warp * 32 + lane; j < listed; j += warps * 32) status[list[j]] = kStFull;
  for (uint32_t j = warp; j < count; j += warps) {
    const uint32_t i = list[j];
    const TableView t = ts.of(i);
    const uint32_t tid = ts.id(i);
    const uint64_t v = load_val(vals, i);
    const Key k = load_key(keys, i);
    const Addr a = address_of(k, t.nb, t.seed);
    const uint8_t st = search_warp<kBfsNodes, kBfsDepth>(t, tid, k, v, a, now, expiry, ws, q, seen);
    if (lane == 0) {
      if (st == kStFull && retry) {
        retry[atomicAdd(retry_count, 1u)] = i;
      } else {
        if (st == kStBusy) latch_error(t, kErrLockTimeout);
        status[i] = st;
      }
    }
  }
}

template <int kBfsNodes>
__host__ __device__ constexpr size_t warp_search_bytes() {
  return kBfsNodes * sizeof(Node) + WarpSeen<kBfsNodes>::kSize * sizeof(uint32_t);
}

template <int kWarps, int kBfsNodes, int kBfsDepth>
__global__ void __launch_bounds__(kWarps * 32, 1) insert_phase2_warp(TableSet ts, const uint8_t* __restrict__ keys,
                                                                  const uint64_t* __restrict__ vals, uint32_t now,
                                                                  uint32_t expiry, uint8_t* __restrict__ status,
                                                                  Workspace ws, const uint32_t* list,
                                                                  const uint32_t* count_ptr, uint32_t* retry,
                                                                  uint32_t* retry_count, uint32_t max_keys) {
  pdl_wait();
  static_assert(kWarps * warp_search_bytes<kBfsNodes>() <= 48 * 1024, "search state exceeds 48 KB");
  __shared__ Node queues[kWarps][kBfsNodes];
  __shared__ uint32_t sets[kWarps][WarpSeen<kBfsNodes>::kSize];
  const uint32_t w = threadIdx.x >> 5;
  phase2_range_warp<kBfsNodes, kBfsDepth>(ts, keys, vals, now, expiry, status, ws, list, ld32_cg(count_ptr), retry,
                                          retry_count, max_keys, queues[w], sets[w], blockIdx.x * kWarps + w,
                                          gridDim.x * kWarps);
}

template <int kThreadsPerBlock, int kBfsNodes, int kBfsDepth>
__global__ void __launch_bounds__(kThreadsPerBlock) insert_phase2(TableSet ts, const uint8_t* __restrict__ keys,
                                                                  const uint64_t* __restrict__ vals, uint32_t now,
                                                                  uint32_t expiry, uint8_t* __restrict__ status,
                                                                  Workspace ws, const uint32_t* list,
                                                                  const uint32_t* count_ptr, uint32_t* retry,
                                                                  uint32_t* retry_count, uint32_t max_keys) {
  pdl_wait();
  static_assert(kThreadsPerBlock * kBfsNodes * sizeof(Node) <= 48 * 1024, "BFS state exceeds 48 KB");
  static_assert(kThreadsPerBlock % 32 == 0 &&
                    (kThreadsPerBlock / 32) * warp_search_bytes<kBfsNodes>() <= kBfsNodes * kThreadsPerBlock * sizeof(Node),
                "the warp form's state does not fit in the queues");
  __shared__ __align__(16) Node queues[kBfsNodes][kThreadsPerBlock];
  const uint32_t listed = ld32_cg(count_ptr);
  if (listed <= kGridWarpKeys) {
    // a short list: one warp per key, each warp's queue and visited set carved from the block's queues
    const uint32_t w = threadIdx.x >> 5;
    uint8_t* mine = reinterpret_cast<uint8_t*>(&queues[0][0]) + w * warp_search_bytes<kBfsNodes>();
    phase2_range_warp<kBfsNodes, kBfsDepth>(ts, keys, vals, now, expiry, status, ws, list, listed, retry,
                                            retry_count, max_keys, reinterpret_cast<Node*>(mine),
                                            reinterpret_cast<uint32_t*>(mine + kBfsNodes * sizeof(Node)),
                                            blockIdx.x * (kThreadsPerBlock / 32) + w,
                                            gridDim.x * (kThreadsPerBlock / 32));
    return;
  }
  const Queue q{&queues[0][threadIdx.x], kThreadsPerBlock};
  phase2_range<kBfsNodes, kBfsDepth>(ts, keys, vals, now, expiry, status, ws, list, listed, retry, retry_count,
                                     max_keys, q, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// ----------------------------------------------------- fixup and finish
// What is left after the last pass, each part a list that is usually short or
// empty: the deferred filter resets, the claimed bits that phase 1 left set in
// timers tables, and the followers (dedup.cuh). The parts touch disjoint words,
// so one launch runs them: filters of buckets whose moved counter is zero; ctrl
// words; the status bytes and stored values of groups with followers.
__device__ void fixup_finish_range(const TableSet& ts, const uint8_t* __restrict__ keys,
                                   const uint64_t* __restrict__ vals, uint8_t* __restrict__ status,
                                   const Workspace& ws, const Counts& counts, uint64_t worker, uint64_t workers) {
  const uint64_t stride = workers;
  const uint64_t i = worker;
  if (counts[kCntFixupOverflow]) {  // the list overflowed: scan every bucket of every table
    for (uint32_t tb = 0; tb < ts.n_tables; ++tb) {
      const TableView t = ts.table(tb);
      for (uint64_t b = i; b < t.nb; b += stride)
        if (ld32_cg(moved_ptr(t, (uint32_t)b)) == 0u) st64_cg(bloom_ptr(t, (uint32_t)b), 0ull);
    }
  } else {
    const uint32_t count = min(counts[kCntFixup], ws.fix_cap);
    for (uint64_t j = i; j < count; j += stride) {
      const unsigned long long e = ws.fixup[j];
      const TableView t = ts.table((uint32_t)(e >> 32));
      const uint32_t b = (uint32_t)e;
      if (ld32_cg(moved_ptr(t, b)) == 0u) st64_cg(bloom_ptr(t, b), 0ull);
    }
  }
  const uint32_t sticky = counts[kCntSticky];
  for (uint64_t j = i; j < sticky; j += stride) {
    const unsigned long long e = ws.sticky[j];
    atomicAnd(ctrl_ptr(ts.of(e >> 32), (uint32_t)e), ~(kBusyMask << kClaimShift));
  }
  const uint32_t followers = counts[kCntFollowers];
  const bool few = followers <= 16384u;
  for (uint64_t j = i; j < followers; j += stride) {
    const uint2 f = ws.followers[j];
    const Key k = load_key(keys, f.x);
    const uint64_t v = load_val(vals, f.x);
    const uint2 range = ws.range[f.y];
    const bool last = f.x > f.y && f.x == range.y;  // its value is the one that stays (y of 0: none above the owner)
    // The buckets of a last occurrence are requested before the owner's outcome is looked at, both
    // at once where there are so few that the time of one counts and not their requests. (Both at
    // once / one after the other: cycles of 32K keys, 90 % of them repeated, 38.3 / 39.7 us; of 256K,
    // 30 %, 82.2 / 81.3, and 1M 251.6 / 247.7.)
    TableView t{};
    Addr a{};
    Snap s1{}, s2{};
    if (last) {
      t = ts.of(f.x);
      a = address_of(k, t.nb, t.seed);
      ld256_cg(bucket_ptr(t, a.b1), s1.w);
      if (few) ld256_cg(bucket_ptr(t, a.b2), s2.w);
    }
    // the owner's outcome; the group's lowest index takes it over (from INSERTED the owner then
    // becomes UPDATED, which every other follower reports for either)
    uint8_t st = *reinterpret_cast<volatile uint8_t*>(status + f.y);
    const bool stored = st == kStInserted || st == kStUpdated;
    if (st == kStInserted && f.x == range.x) {
      status[f.y] = kStUpdated;
    } else if (stored) {
      st = kStUpdated;  // FULL and BUSY copy through
    }
    status[f.x] = st;
    if (last && stored) {
      const int in1 = find_key(t, a.b1, (uint32_t)s1.w[3], s1, k, a.tag);
      if (in1 < 0 && !few) ld256_cg(bucket_ptr(t, a.b2), s2.w);
      const int in2 = in1 >= 0 ? -1 : find_key(t, a.b2, (uint32_t)s2.w[3], s2, k, a.tag);
      if (in1 >= 0) st64_cg(value_ptr(t, a.b1, in1), v);
      if (in2 >= 0) st64_cg(value_ptr(t, a.b2, in2), v);
    }
  }
}

__global__ void __launch_bounds__(kThreads) insert_fixup_finish(TableSet ts, const uint8_t* __restrict__ keys,
                                                                const uint64_t* __restrict__ vals,
                                                                uint8_t* __restrict__ status, Workspace ws) {
  pdl_wait();
  fixup_finish_range(ts, keys, vals, status, ws, load_counts(ws), blockIdx.x * (uint64_t)blockDim.x + threadIdx.x,
                     (uint64_t)gridDim.x * blockDim.x);
}

// What a small batch's cluster leaves (insert_cluster<false> below): the searches of the
// keys that the one-move pass could not place, one warp per key, each going on to
// the next width by itself, and then, in the last block to finish, the finishing
// pass. A launch of its own because the widest search takes 50 us if it fails and
// a cluster has room for few at a time: 256 keys bound for a full table take 0.1
// ms by these two launches, 12.7 ms when the cluster ran all passes, 0.12 ms as a
// chain; 2048 keys 0.21, 6.6 and 0.19 ms. It costs batches that leave nothing 1.2
// to 1.6 us.
constexpr unsigned kRestBlocksPerSm = 6;  // 32 KB of queue and visited set each
constexpr int kRestThreads = 128;  // one warp searches, all take part in the finishing pass
__global__ void __launch_bounds__(kRestThreads) insert_rest(TableSet ts, const uint8_t* __restrict__ keys,
                                                            const uint64_t* __restrict__ vals, uint32_t now,
                                                            uint32_t expiry, uint8_t* __restrict__ status,
                                                            Workspace ws) {
  __shared__ Node queue[2048];
  __shared__ uint32_t seen[WarpSeen<2048>::kSize];
  __shared__ bool last;
  pdl_wait();
  const uint32_t listed = ld32_cg(ws.counters + kCntMoved1), blocks = min(gridDim.x, listed);
  if (blockIdx.x >= blocks) return;
  if (threadIdx.x < 32) {
    for (uint32_t j = blockIdx.x; j < listed; j += blocks) {
      const uint32_t i = ws.retry[j];
      const TableView t = ts.of(i);
      const uint32_t tid = ts.id(i);
      const uint64_t v = load_val(vals, i);
      const Key k = load_key(keys, i);
      const Addr a = address_of(k, t.nb, t.seed);
      uint8_t st = search_warp<96, 4>(t, tid, k, v, a, now, expiry, ws, queue, seen);
      if (st == kStFull) {
        if (threadIdx.x == 0) atomicAdd(ws.counters + kCntGrid, 1u);
        st = search_warp<192, 5>(t, tid, k, v, a, now, expiry, ws, queue, seen);
      }
      if (st == kStFull) {
        uint32_t taken = 0;
        if (threadIdx.x == 0) taken = atomicAdd(ws.counters + kCntSecond, 1u);
        if (__shfl_sync(kWarpAll, taken, 0) < kLastPassKeys)
          st = search_warp<2048, 6>(t, tid, k, v, a, now, expiry, ws, queue, seen);
      }
      if (threadIdx.x == 0) {
        if (st == kStBusy) latch_error(t, kErrLockTimeout);
        status[i] = st;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    fence_acq_rel();
    last = atomicAdd(ws.counters + kCntRest, 1u) == blocks - 1;
    fence_acq_rel();
  }
  __syncthreads();
  if (last) fixup_finish_range(ts, keys, vals, status, ws, load_counts(ws), threadIdx.x, kRestThreads);
}

// --------------------------------------------------------- small batches
// The stages of the chain above on one cluster, in order, with a cluster barrier
// between them instead of a kernel boundary: a small batch spends most of a
// chain's time in the starts and drains of its seven dependent launches, each
// also 1.9 us of host time, and a cluster's barrier takes a fraction of either. A
// stage whose list is empty is skipped with its barrier. Two forms:
//   whole (at most 64 keys)  eight blocks of one cluster run the whole call. The
//         first one works alone until there are keys without a slot, with the set
//         and the groups of equal keys in shared memory (an update of 64 keys 5.7
//         us, 6.4 with the set in the workspace and all blocks at work); the
//         others are there for the searches, 48 of the widest at a time;
//   first (up to 2048 keys)  one cluster of up to eight blocks runs the stages up
//         to the one-move pass, and the finishing pass if that leaves nothing;
//         insert_rest, launched after it, the rest. A batch that fits one block
//         has one, with the set and the groups in shared memory.
// The whole form's search queues take the place of phase 1's shared memory: the
// grid and the second pass run on every warp (96 and 192 nodes and a visited set
// each), the last (2048 nodes and the visited set) on six warps of every block.
// The largest batch of the whole form: 64 keys bound for a full table, two rounds
// of the widest search, take 150 us, a chain 115; 32 keys 104 and 114.
constexpr uint64_t kWholeKeys = 64;
constexpr unsigned kWholeBlocks = 8;
constexpr uint32_t kWholeWidest = 6;  // warps of a block that run the last pass
constexpr int kClusterThreads = 256;
// Shared memory: phase 1's rows and lists, then the set; the queues over both; the
// groups, which the finishing pass reads, behind.
constexpr size_t kOneSetAt = 20 * 1024;
constexpr size_t kFirstGroupsAt = kOneSetAt + sizeof(OneBlockSet);
constexpr size_t kFirstSmem = kFirstGroupsAt + sizeof(OneBlockGroups);
constexpr size_t kWholeGroupsAt = kWholeWidest * warp_search_bytes<2048>();
constexpr size_t kWholeSmem = kWholeGroupsAt + sizeof(OneBlockGroups);
static_assert((kClusterThreads / 32) * sizeof(P1Rows) + sizeof(P1Lists) <= kOneSetAt && kFirstSmem <= 48 * 1024 &&
                  kFirstGroupsAt <= kWholeGroupsAt &&
                  (kClusterThreads / 32) * warp_search_bytes<192>() <= kWholeGroupsAt &&
                  (kClusterThreads / 32) * warp_search_bytes<96>() <= kWholeGroupsAt,
              "the parts of the shared memory overlap");
static_assert(kOneBlockKeys == kClusterThreads, "cluster_blocks gives batches that fit one block a cluster of one");
static_assert(kWholeKeys <= kOneBlockKeys, "a whole form's batch fits its first block");

template <bool kWhole, bool kTimers>
__global__ void __launch_bounds__(kClusterThreads, kWhole ? 1 : 2)
    insert_cluster(TableSet ts, const uint8_t* __restrict__ keys, const uint64_t* __restrict__ vals, uint64_t n,
                   uint32_t now, uint32_t expiry, uint8_t* __restrict__ status, Workspace caller_ws) {
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t tid = blockIdx.x * kClusterThreads + threadIdx.x;
  const uint32_t threads = gridDim.x * kClusterThreads;
  // the threads that share phase 1 and the finishing pass: one block's or all
  const bool one = kWhole || gridDim.x == 1;
  const uint32_t own_threads = one ? kClusterThreads : threads;
  const Workspace ws = one ? in_shared(caller_ws, *reinterpret_cast<OneBlockSet*>(smem + kOneSetAt),
                                       *reinterpret_cast<OneBlockGroups*>(smem + (kWhole ? kWholeGroupsAt : kFirstGroupsAt)))
                           : caller_ws;
  pdl_wait();
  if (!kWhole || blockIdx.x == 0) {
    clear_workspace(ws, tid, own_threads);
    if (kWhole) {
      __syncthreads();
    } else {
      cluster_barrier();
    }
    P1Rows* rows = reinterpret_cast<P1Rows*>(smem);
    P1Lists& lists = *reinterpret_cast<P1Lists*>(rows + kClusterThreads / 32);
    lists_init(lists);
    for (uint64_t first = blockIdx.x * (uint64_t)kClusterThreads; first < n; first += own_threads) {  // whole blocks
      const uint64_t i = first + threadIdx.x;
      phase1_one<kTimers>(ts, keys, vals, now, expiry, status, ws, i, i < n, rows[threadIdx.x >> 5], lists);
    }
  }
  cluster_barrier();
  // lists as in the chain: pending -> one move -> retry -> grid search -> pending -> second pass ->
  // retry -> last pass. A pass whose list is empty is skipped with its barrier, and so are the ones
  // after it; every block reads the same counts (final before the barrier), so all skip alike.
  Counts counts = load_counts(ws);
  if (counts[kCntPending]) {
    if (counts[kCntPending] <= threads / 16u) {
      move1_range_half(ts, keys, vals, now, expiry, status, ws, ws.pending, counts[kCntPending], ws.retry,
                       ws.counters + kCntMoved1, tid / 16u, threads / 16u);
    } else {
      move1_range(ts, keys, vals, now, expiry, status, ws, ws.pending, counts[kCntPending], ws.retry,
                  ws.counters + kCntMoved1, tid, threads);
    }
    cluster_barrier();
    counts = load_counts(ws);
  }
  if constexpr (!kWhole) {
    if (counts[kCntMoved1]) {  // insert_rest goes on from here
      if (one) {
        for (uint32_t j = threadIdx.x; j < ws.n; j += kClusterThreads) caller_ws.range[j] = ws.range[j];
        for (uint32_t j = threadIdx.x; j < counts[kCntFollowers]; j += kClusterThreads)
          caller_ws.followers[j] = ws.followers[j];
      }
      return;
    }
    fixup_finish_range(ts, keys, vals, status, ws, counts, tid, own_threads);
  } else {
    const uint32_t w = threadIdx.x >> 5, warp = blockIdx.x * (kClusterThreads / 32) + w;
    const uint32_t warps = gridDim.x * (kClusterThreads / 32);
    if (const uint32_t listed = counts[kCntMoved1]) {
      uint8_t* mine = smem + w * warp_search_bytes<96>();
      phase2_range_warp<96, 4>(ts, keys, vals, now, expiry, status, ws, ws.retry, listed, ws.pending,
                               ws.counters + kCntGrid, 0xFFFFFFFFu, reinterpret_cast<Node*>(mine),
                               reinterpret_cast<uint32_t*>(mine + 96 * sizeof(Node)), warp, warps);
      cluster_barrier();
      counts = load_counts(ws);
    }
    if (const uint32_t listed = counts[kCntGrid]) {
      uint8_t* mine = smem + w * warp_search_bytes<192>();
      phase2_range_warp<192, 5>(ts, keys, vals, now, expiry, status, ws, ws.pending, listed, ws.retry,
                                ws.counters + kCntSecond, kSecondPassKeys, reinterpret_cast<Node*>(mine),
                                reinterpret_cast<uint32_t*>(mine + 192 * sizeof(Node)), warp, warps);
      cluster_barrier();
      counts = load_counts(ws);
    }
    if (const uint32_t listed = counts[kCntSecond]) {
      uint8_t* mine = smem + w * warp_search_bytes<2048>();
      if (w < kWholeWidest)  // the first keys to different blocks
        phase2_range_warp<2048, 6>(ts, keys, vals, now, expiry, status, ws, ws.retry, listed, (uint32_t*)nullptr,
                                   (uint32_t*)nullptr, kLastPassKeys, reinterpret_cast<Node*>(mine),
                                   reinterpret_cast<uint32_t*>(mine + 2048 * sizeof(Node)), w * gridDim.x + blockIdx.x,
                                   kWholeWidest * gridDim.x);
      cluster_barrier();
      counts = load_counts(ws);
    }
    if (blockIdx.x == 0) fixup_finish_range(ts, keys, vals, status, ws, counts, tid, own_threads);
  }
}

// ------------------------------------------------------- workspace reset
__global__ void __launch_bounds__(kThreads) workspace_clear(Workspace ws) {
  pdl_wait();
  clear_workspace(ws, blockIdx.x * kThreads + threadIdx.x, gridDim.x * kThreads);
}

}  // namespace

cudaError_t launch_workspace_clear(const Workspace& ws, cudaStream_t s) {
  // m is a power of two >= 64 and the set is 256-byte aligned: whole 16-byte vectors
  const uint64_t n_vec = ((uint64_t)ws.m_mask + 1) / 4;
  const uint64_t want = n_vec > kCounterWords ? n_vec : kCounterWords;
  const uint64_t blocks = (want + kThreads - 1) / kThreads;
  const uint64_t cap = 16ull * device_sm_count();
  return launch_chained(workspace_clear, (unsigned)(blocks < cap ? blocks : cap), kThreads, s, ws);
}

namespace {

// kInsertLaunchSingle, once meant for a cooperative launch of the whole call, runs the
// chain whatever the batch's size.
std::atomic<int> g_insert_launch{kInsertLaunchChain};

// Allows the whole cluster's shared memory, once per device.
cudaError_t allow_whole_cluster() {
  constexpr int kMaxDevices = 64;
  static std::atomic<bool> done[kMaxDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev >= 0 && dev < kMaxDevices;
  if (known && done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  if ((e = cudaFuncSetAttribute(insert_cluster<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kWholeSmem)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(insert_cluster<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kWholeSmem)) != cudaSuccess)
    return e;
  if (known) done[dev].store(true, std::memory_order_relaxed);
  return cudaSuccess;
}

}  // namespace

int set_insert_launch(int mode) {
  if (mode != kInsertLaunchChain && mode != kInsertLaunchSingle) return -1;
  return g_insert_launch.exchange(mode);
}

cudaError_t launch_insert(const TableSet& ts, const uint8_t* keys, const uint64_t* vals, uint64_t n, uint32_t now,
                          uint32_t expiry, uint8_t* status, const Workspace& ws, cudaStream_t s) {
  cudaError_t e;
  if (n <= kClusterKeys && g_insert_launch.load(std::memory_order_relaxed) != kInsertLaunchSingle) {
    if (n <= kWholeKeys) {
      if ((e = allow_whole_cluster()) != cudaSuccess) return e;
      return launch_cluster(ts.any_timers ? insert_cluster<true, true> : insert_cluster<true, false>, kWholeBlocks,
                            kClusterThreads, kWholeSmem, s, ts, keys, vals, n, now, expiry, status, ws);
    }
    e = launch_cluster(ts.any_timers ? insert_cluster<false, true> : insert_cluster<false, false>,
                       cluster_blocks(n, kClusterThreads), kClusterThreads, kFirstSmem, s, ts, keys, vals, n, now, expiry,
                       status, ws);
    if (e != cudaSuccess) return e;
    const unsigned most = kRestBlocksPerSm * (unsigned)device_sm_count();
    return launch_chained(insert_rest, n < most ? (unsigned)n : most, kRestThreads, s, ts, keys, vals, now, expiry, status,
                          ws);
  }
  e = launch_workspace_clear(ws, s);
  if (e != cudaSuccess) return e;
  const unsigned sms = (unsigned)device_sm_count();
  e = launch_chained(ts.any_timers ? insert_phase1<true> : insert_phase1<false>, grid_for(n, kP1Threads), kP1Threads, s, ts,
                     keys, vals, n, now, expiry, status, ws);
  if (e != cudaSuccess) return e;
  // lists: phase 1 -> pending [0] -> move1 -> retry [3] -> grid search ->
  // pending [5] -> second search -> retry [6] -> last search
  // each pass's list holds at most n keys: no more blocks than that many keys can use
  const auto cap = [n](unsigned blocks, unsigned keys_per_block) {
    const uint64_t want = (n + keys_per_block - 1) / keys_per_block;
    return want < blocks ? (unsigned)want : blocks;
  };
  const unsigned by_thread = cap(sms * 16, kThreads), by_half = cap(kMoveHalfKeys / (kThreads / 16), kThreads / 16);
  e = launch_chained(insert_move1, by_thread > by_half ? by_thread : by_half, kThreads, s, ts, keys, vals, now, expiry, status, ws,
                     (const uint32_t*)ws.pending, (const uint32_t*)(ws.counters + kCntPending), ws.retry, ws.counters + kCntMoved1);
  if (e != cudaSuccess) return e;
  e = launch_chained(insert_phase2<kP2Threads, 96, 4>, cap(sms * 4, kP2Threads / 32), kP2Threads, s, ts, keys, vals, now, expiry, status,
                     ws, (const uint32_t*)ws.retry, (const uint32_t*)(ws.counters + kCntMoved1), ws.pending, ws.counters + kCntGrid,
                     0xFFFFFFFFu);
  if (e != cudaSuccess) return e;
  // second pass, one warp per key: the keys the grid pass could not place
  e = launch_chained(insert_phase2_warp<8, 192, 5>, cap(sms * 2, 8), 8 * 32, s, ts, keys, vals, now, expiry, status, ws,
                     (const uint32_t*)ws.pending, (const uint32_t*)(ws.counters + kCntGrid), ws.retry, ws.counters + kCntSecond,
                     kSecondPassKeys);
  if (e != cudaSuccess) return e;
  // last pass, one warp per key: the widest search; a key is FULL only if it finds no path
  e = launch_chained(insert_phase2_warp<1, 2048, 6>, cap(kLastPassKeys, 1), 32, s, ts, keys, vals, now, expiry, status, ws,
                     (const uint32_t*)ws.retry, (const uint32_t*)(ws.counters + kCntSecond), (uint32_t*)nullptr,
                     (uint32_t*)nullptr, kLastPassKeys);
  if (e != cudaSuccess) return e;
  // Two blocks per SM, and from 256K keys one thread to four keys: how many followers there are is not
  // known here, and a chain of four dependent reads for each wants more of them in flight (1M keys into
  // 16M buckets, 30 % of them repeated, all present: 140.4 us with two blocks, 132.2 with these; none
  // repeated: 126.2 and 127.5; 128K keys gain nothing from more than two).
  const unsigned fin_least = cap(sms * 2, kThreads), fin_most = cap(sms * 8, kThreads * 4);
  return launch_chained(insert_fixup_finish, fin_most > fin_least ? fin_most : fin_least, kThreads, s, ts, keys, vals,
                        status, ws);
}

}  // namespace ckpp
