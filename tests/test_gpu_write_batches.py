"""Insert and delete batches against the CPU oracle at the sizes where their
kernels change shape (warps, blocks, tiles, the small and the large form), with
every kind of key in one batch: new ones, stored ones, ones whose entry is dead,
and repeated ones, among them one that makes up a quarter of the batch."""

import numpy as np
import pytest
import torch

import oracle
from gpu_layout import download, oracle_live
from paper_1712_09624_gb300 import workload as W

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 33, 255, 257, 511, 513, 1025, 4095, 4097, 8191, 8193, 16385, 32769, 70001]


def mixed_batch(rng, pool, n):
    """n keys of the pool: a quarter are one key, the rest uniform with repeats."""
    i = rng.integers(0, pool.shape[0], n)
    i[rng.random(n) < 0.25] = rng.integers(0, pool.shape[0])
    return pool[i]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("timers", [False, True])
def test_write_batches_match_the_oracle(n, timers):
    from paper_1712_09624_gb300.table import FlowTable
    nb = max(16, n // 4)
    rng = np.random.default_rng(1000 + n)
    pool = W.make_keys(300 + n, 70, int(0.8 * nb * 8))
    g, o = FlowTable(nb, timers=timers, seed=n), oracle.Table(nb, 8, timers, n)
    now = 20
    for step in range(4):
        keys = mixed_batch(rng, pool, n)
        vals = rng.integers(0, 2**63, n, dtype=np.int64).astype(np.uint64)
        ttl = [5, 900, 30, 1][step] if timers else 0
        assert (g.insert(keys, vals, now, ttl).cpu().numpy() == o.insert(keys, vals, now, ttl)).all(), step
        d = download(g)
        assert d.check() == [] and d.live(now) == oracle_live(o, now), step
        if timers:
            now += 7  # some of the entries are dead from here on
        keys = mixed_batch(rng, pool, n)
        assert (g.delete(keys, now).cpu().numpy() == o.delete(keys, now)).all(), step
        d = download(g)
        assert d.check() == [] and d.live(now) == oracle_live(o, now), step
        q = W.make_keys(9, 71, 50)
        gv, gf = g.lookup(np.concatenate([pool, q]), now)
        ov, of = o.lookup(np.concatenate([pool, q]), now)
        assert (gf.cpu().numpy() == of).all() and (gv.cpu().numpy().view(np.uint64) == ov).all()
    assert g.sync_status() == 0


@pytest.mark.parametrize("n", [1, 257, 4097, 70001])
def test_write_batches_over_tables_with_and_without_timers(n):
    """The multi-table calls on one batch for tables of both layouts, the same key
    bound for several of them, and indices that name no table."""
    from paper_1712_09624_gb300 import _ckpp as K
    from paper_1712_09624_gb300.batched import BatchedLookup
    from paper_1712_09624_gb300.table import FlowTable
    nb = max(16, n // 8)
    rng = np.random.default_rng(2000 + n)
    kinds = [False, True, False, True]
    tables = [FlowTable(nb + t, timers=k, seed=5) for t, k in enumerate(kinds)]
    oracles = [oracle.Table(nb + t, 8, k, 5) for t, k in enumerate(kinds)]
    batch = BatchedLookup(tables, max_jobs=1)
    pool = W.make_keys(400 + n, 72, int(0.7 * nb * 8))
    ws = torch.empty(K.ckpp_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    now = 50
    for step in range(3):
        keys = mixed_batch(rng, pool, n)
        ids = rng.integers(0, len(kinds) + 1, n).astype(np.int32)  # the last names no table
        vals = rng.integers(0, 2**62, n)
        dk, di = torch.from_numpy(np.ascontiguousarray(keys)).cuda(), torch.from_numpy(ids).cuda()
        st = torch.empty(n, dtype=torch.uint8, device="cuda")
        K.ckpp_batch_insert(batch.handle, dk, di, torch.from_numpy(vals).cuda(), st, ws, now, 40)
        got = st.cpu().numpy()
        want = np.full(n, K.ST_NO_TABLE, np.uint8)
        for t, o in enumerate(oracles):
            sel = ids == t
            if sel.any():
                want[sel] = o.insert(keys[sel], vals[sel].astype(np.uint64), now, 40 if kinds[t] else 0)
        assert (got == want).all(), step
        now += 30 * step
        part = rng.random(n) < 0.5
        m = int(part.sum())
        if m:
            K.ckpp_batch_delete(batch.handle, dk[torch.from_numpy(part).cuda()].contiguous(),
                                di[torch.from_numpy(part).cuda()].contiguous(), st[:m], ws, now)
            want = np.full(m, K.ST_NO_TABLE, np.uint8)
            for t, o in enumerate(oracles):
                sel = ids[part] == t
                if sel.any():
                    want[sel] = o.delete(keys[part][sel], now)
            assert (st[:m].cpu().numpy() == want).all(), step
        for t, o in enumerate(oracles):
            d = download(tables[t])
            assert d.check() == [] and d.live(now) == oracle_live(o, now), (step, t)
