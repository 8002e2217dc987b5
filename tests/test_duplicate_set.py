"""The set in which a write batch finds its equal keys, filled on the host by the
device code: how many occupied positions a key passes and how many other keys it
reads, whatever the batch's keys have in common: one shard (bits 16-31 of the
primary hash), one tag (bits 0-15), one region of buckets (the top bits)."""

import ctypes as C

import numpy as np
import pytest

import host_model as H

ACCESS = """
constexpr uint32_t kNoIndex = 0xFFFFFFFFu;
struct Workspace { uint32_t* set; uint32_t m_mask, idx_bits; };
struct TableSet { const uint32_t* tab; uint32_t id(uint64_t i) const { return tab[i]; } };
static uint64_t steps, reads;
static uint32_t atomicCAS(uint32_t* p, uint32_t want, uint32_t to) {
  ++steps;
  const uint32_t old = *p;
  if (old == want) *p = to;
  return old;
}
static Key load_key(const uint8_t* keys, uint64_t i) {
  ++reads;
  const uint64_t* k = (const uint64_t*)(keys + 16 * i);
  return Key{k[0], k[1]};
}
"""

DRIVER = """
extern "C" void fill(uint32_t* set, uint32_t m_mask, uint32_t idx_bits, const uint8_t* keys, const uint64_t* h1,
                     const uint32_t* tab, uint64_t n, uint32_t* owner, uint64_t* counts) {
  const Workspace ws{set, m_mask, idx_bits};
  const TableSet ts{tab};
  steps = reads = 0;
  for (uint64_t i = 0; i < n; ++i) {
    const uint64_t* k = (const uint64_t*)(keys + 16 * i);
    owner[i] = set_owner(ws, ts, keys, Key{k[0], k[1]}, tab[i], (uint32_t)i, set_probe(ws, h1[i], tab[i], (uint32_t)i));
  }
  counts[0] = steps, counts[1] = reads;
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    code = H.layout() + ACCESS + H.definitions("dedup.cuh", "SetProbe", "set_probe", "set_owner") + DRIVER
    return C.CDLL(H.build(tmp_path_factory.mktemp("set"), code))


def fill(model, keys, h1, tab):
    """Owners, steps and key reads of a batch, with the set sized as ws_layout (api_internal.h) sizes it."""
    n, m = h1.shape[0], 64
    while m < (8 * n if n <= 1 << 17 else 4 * n):
        m *= 2
    words, owner, counts = np.full(m, 0xFFFFFFFF, np.uint32), np.empty(n, np.uint32), np.zeros(2, np.uint64)
    p = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    model.fill(p(words), C.c_uint32(m - 1), C.c_uint32(n.bit_length()), p(keys), p(h1), p(tab), C.c_uint64(n), p(owner),
               p(counts))
    return owner, int(counts[0]), int(counts[1]), n / m


# bits of the primary hash that all keys of the batch share
COMMON = {"none": 0, "one of 8 shards": 0x7 << 29, "one of 64 shards": 0x3F << 26, "all of the shard's bits": 0xFFFF << 16,
          "a tag": 0xFFFF, "a region of buckets": 0xFF << 56, "a shard and a region": 0x3F << 26 | 0xFF << 56}


@pytest.mark.parametrize("common", COMMON)
@pytest.mark.parametrize("n", [2048, 32768, 1 << 17, 1 << 20])
def test_few_positions_are_passed_and_hardly_a_key_is_read(model, n, common):
    rng = np.random.default_rng(n)
    h1 = rng.integers(0, 2**64, n, dtype=np.uint64)
    fixed = np.uint64(COMMON[common])
    h1 = (h1 & ~fixed) | (rng.integers(0, 2**64, dtype=np.uint64) & fixed)
    keys = np.stack([h1, np.arange(n, dtype=np.uint64)], axis=1)  # distinct
    owner, steps, reads, load = fill(model, keys, h1, np.zeros(n, np.uint32))
    assert (owner == np.arange(n)).all()
    # linear probing at this load (Knuth, vol. 3, 6.4); a word keeps 32 - bit_length(n) hash bits
    passed = 0.5 * (1 / (1 - load) - 1)
    assert steps / n - 1 <= 1.25 * passed + 0.02
    assert reads / n <= 2 * passed / 2.0 ** (32 - n.bit_length()) + 0.002


def test_equal_keys_of_a_table_have_one_owner(model):
    rng = np.random.default_rng(5)
    n = 20_000
    which = np.where(rng.random(n) < 0.3, 0, rng.integers(0, 4000, n))  # one key makes up a third
    h1 = rng.integers(0, 2**64, 4000, dtype=np.uint64)[which]
    keys = np.stack([which.astype(np.uint64), np.zeros(n, np.uint64)], axis=1)
    tab = rng.integers(0, 3, n).astype(np.uint32)
    owner, *_ = fill(model, keys, h1, tab)
    group = which * 3 + tab
    first = {g: i for i, g in reversed(list(enumerate(group.tolist())))}
    assert (owner == [first[g] for g in group.tolist()]).all()
