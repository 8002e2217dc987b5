"""What an insert does in a bucket while another key of the batch takes a slot of
it, for every order in which that key's stores can become visible: the entry's
words lie in different lines, so nothing orders them; only the claim comes first,
and the publication of a slot that was free last (a slot that held a dead entry
stays busy, with its claim, and has none)."""

import ctypes as C
import itertools

import pytest

import host_model as H

# Memory accesses of the model. Time passes with every access of the key that is
# watched. The other key's claim, its entry's key and expiry, and its publication
# become visible at times of their own (ev[0..3]); cas_fails: every CAS finds its
# word changed.
ACCESS = """
static uint8_t bucket_mem[256];
static int clock_now, ev[4], cas_fails, latched, was_free;
static uint32_t ctrl0, slot, expiry_of_batch;
static uint64_t other_key[2];
static void tick();
static void fence_acq_rel() {}
static void ld128_cg(const void* p, uint64_t& a, uint64_t& b) {
  tick();
  a = ((const uint64_t*)p)[0], b = ((const uint64_t*)p)[1];
}
static uint32_t ld32_cg(const void* p) { tick(); return *(const uint32_t*)p; }
static uint32_t atomicCAS(uint32_t* p, uint32_t want, uint32_t to) {
  tick();
  if (cas_fails) return want ^ (1u << 30);
  const uint32_t old = *p;
  if (old == want) *p = to;
  return old;
}
struct Snap { uint64_t w[4]; uint64_t e0, e1; };
static void latch_error(const TableView&, uint32_t) { ++latched; }
"""

DRIVER = """
static TableView view() { return TableView{bucket_mem, nullptr, 16, 0, 1, 0}; }
static void put_key(uint32_t s, uint64_t a, uint64_t b) {
  uint64_t* k = (uint64_t*)(bucket_mem + key_off(1, s));
  k[0] = a, k[1] = b;
}
static void put_expiry(uint32_t s, uint32_t e) { ((uint16_t*)(bucket_mem + kExpiryOff))[s] = (uint16_t)e; }
static void tick() {
  const int t = clock_now++;
  uint32_t* ctrl = (uint32_t*)(bucket_mem + 24);
  if (t == ev[0]) *ctrl |= claim_bit(slot);
  if (t == ev[1]) put_key(slot, other_key[0], other_key[1]);
  if (t == ev[2]) put_expiry(slot, expiry_of_batch);
  if (t == ev[3] && was_free) *ctrl ^= claim_bit(slot) | 1u << slot;
}
static void start(uint32_t busy, uint32_t expiry, const int* at) {
  for (int i = 0; i < 256; ++i) bucket_mem[i] = 0;
  *(uint32_t*)(bucket_mem + 24) = busy;
  clock_now = cas_fails = latched = was_free = 0;
  expiry_of_batch = expiry;
  other_key[0] = 77, other_key[1] = 78;
  for (int i = 0; i < 4; ++i) ev[i] = at[i];
}
static Snap snapshot(int expiries_first) {
  Snap s;
  const uint64_t* w = (const uint64_t*)bucket_mem;
  for (int i = 0; i < 2; ++i) {
    tick();
    if ((i == 0) == (expiries_first != 0)) s.e0 = w[4], s.e1 = w[5];
    else for (int j = 0; j < 4; ++j) s.w[j] = w[j];
  }
  return s;
}
// The key has an entry in slot `mine` with expiry `stored`; the other key takes slot
// `taken`, whose entry is dead. expiries_first: which of the snapshot's reads comes first.
// Returns the status (0: the key has to look for a slot), or -1 if the key was not found.
extern "C" int stored(uint32_t mine, uint32_t taken, uint32_t stored_expiry, uint32_t now, uint32_t expiry,
                      int expiries_first, int as_secondary, const int* at) {
  start(1u << mine | 1u << taken, expiry, at);
  slot = taken;
  const Key k{5, 6};
  const uint32_t tag = 9;
  put_key(taken, 7, 8);
  put_expiry(taken, now - 20);
  put_key(mine, k.k0, k.k1);
  put_expiry(mine, stored_expiry);
  ((uint16_t*)bucket_mem)[mine] = (uint16_t)tag;
  const Snap s = snapshot(expiries_first);
  const TableView t = view();
  P1Bucket r = p1_bucket(0, s, tag, true, now, expiry), none{};
  bool second;
  const int sl = as_secondary ? p1_search(t, none, r, k, now, expiry, second) : p1_search(t, r, none, k, now, expiry, second);
  P1Work work = kP1None;
  const int st = sl < 0 ? -1 : p1_stored(t, r, (uint32_t)sl, true, work);
  return st;
}
// The key is not stored, and slot `taken` is the only one that it could claim: free, or
// with a dead entry. Returns whether it claimed the slot after the other key had.
extern "C" int claimed_twice(uint32_t taken, int free, uint32_t now, uint32_t expiry, int expiries_first,
                             int as_secondary, const int* at) {
  start(free ? 0xFFu & ~(1u << taken) : 0xFFu, expiry, at);
  slot = taken;
  was_free = free;
  for (uint32_t s = 0; s < 8; ++s) put_expiry(s, s == taken ? now - 20 : now + 3);
  const Snap s = snapshot(expiries_first);
  const TableView t = view();
  P1Bucket r = p1_bucket(0, s, 9, true, now, expiry), none{};
  bool second;
  if (as_secondary) p1_search(t, none, r, Key{5, 6}, now, expiry, second);
  else p1_search(t, r, none, Key{5, 6}, now, expiry, second);
  uint32_t prev = 0;
  const int got = claim_slot(t, r, false, prev);
  return got >= 0 && clock_now > at[0];
}
extern "C" int lost_claim(int revival) {
  const int never[4] = {-1, -1, -1, -1};
  start(revival ? 1u : 0u, 0, never);
  cas_fails = 1;
  P1Bucket r{};
  r.ctrl = revival ? 1u : 0u;
  r.dead = r.ctrl;
  P1Work work = kP1None;
  uint32_t prev = 0;
  const TableView t = view();
  const int got = revival ? p1_stored(t, r, 0, true, work) : claim_slot(t, r, false, prev);
  return latched == 1 ? got : 1000 + latched;
}
"""

NOW, EXPIRY = 1000, 1040
INSERTED, UPDATED, BUSY = 1, 2, 6


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    code = (H.layout() + ACCESS + "constexpr int kClaimAttempts = 64;\n" +
            H.definitions("insert.cu", "claim_bit", "claimable", "P1Bucket", "p1_expiries", "p1_bucket", "p1_find", "p1_search", "claim_revival",
                          "P1Work", "p1_stored", "claim_slot") + DRIVER)
    return C.CDLL(H.build(tmp_path_factory.mktemp("claims"), code))


def schedules():
    """(claim, key, expiry, publication): the claim first, the publication last, between them any order."""
    for claim in range(9):
        for key, expiry in itertools.product(range(claim, 9), repeat=2):
            for publication in range(max(key, expiry), 9):
                yield claim, key, expiry, publication


def outcome(model, mine, taken, expiry, first, secondary, at):
    return model.stored(mine, taken, expiry, NOW, EXPIRY, first, secondary, (C.c_int * 4)(*at))


@pytest.mark.parametrize("secondary", [0, 1])
@pytest.mark.parametrize("expiries_first", [0, 1])
def test_a_dead_entry_whose_slot_is_taken_is_never_updated_in_place(model, expiries_first, secondary):
    for at in schedules():
        for slot in (0, 5):  # its entry in the bucket's first and second line
            assert outcome(model, slot, slot, NOW - 20, expiries_first, secondary, at) in (-1, 0, INSERTED), at


@pytest.mark.parametrize("secondary", [0, 1])
@pytest.mark.parametrize("expiries_first", [0, 1])
@pytest.mark.parametrize("expiry", [NOW, EXPIRY, EXPIRY + 5])
def test_a_live_entry_is_updated_in_place_whatever_the_rest_of_its_bucket_does(model, expiry, expiries_first, secondary):
    for at in schedules():
        for mine, taken in ((0, 5), (5, 0), (2, 3)):
            assert outcome(model, mine, taken, expiry, expiries_first, secondary, at) == UPDATED, at


@pytest.mark.parametrize("secondary", [0, 1])
@pytest.mark.parametrize("expiries_first", [0, 1])
@pytest.mark.parametrize("free", [0, 1])
def test_a_slot_is_claimed_once(model, free, expiries_first, secondary):
    for at in schedules():
        for slot in (0, 5):
            assert not model.claimed_twice(slot, free, NOW, EXPIRY, expiries_first, secondary, (C.c_int * 4)(*at)), at


def test_a_claim_that_gives_up_latches_the_error(model):
    assert model.lost_claim(1) == BUSY
    assert model.lost_claim(0) == -2
