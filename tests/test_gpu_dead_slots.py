"""Inserts into timers tables whose buckets are full of dead entries: half of the
batch's keys have a dead entry of their own (revived, or inserted anew where another
key has taken its slot), half are new and take dead slots, some keys are repeated."""

import numpy as np
import pytest

import oracle
from gpu_layout import download, oracle_live
from paper_1712_09624_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [60, 2000, 40_000, 1 << 20])
def test_dead_entries_are_revived_and_their_slots_reused(n):
    from paper_1712_09624_gb300.table import FlowTable
    nb = max(16, n // 6)  # a batch fills three quarters of the slots that hold dead entries
    rng = np.random.default_rng(5000 + n)
    g, o = FlowTable(nb, timers=True, seed=n), oracle.Table(nb, 8, True, n)
    own = W.make_keys(1100 + n, 77, int(0.9 * nb * 8))
    now = 5
    for step in range(3):
        vals = rng.integers(0, 2**62, own.shape[0]).astype(np.uint64)
        assert (g.insert(own, vals, now, 3).cpu().numpy() == o.insert(own, vals, now, 3)).all(), step
        now += 10  # every entry is dead
        fresh = W.make_keys(1200 + n + step, 78, n)
        keys = np.where((rng.random(n) < 0.5)[:, None], own[rng.integers(0, own.shape[0], n)], fresh)
        vals = rng.integers(0, 2**62, n).astype(np.uint64)
        assert (g.insert(keys, vals, now, 900).cpu().numpy() == o.insert(keys, vals, now, 900)).all(), step
        d = download(g)
        assert d.check() == [] and d.live(now) == oracle_live(o, now), step
        q = np.concatenate([keys, own])
        v, f = g.lookup(q, now)
        ov, of = o.lookup(q, now)
        assert (f.cpu().numpy() == of).all() and (v.cpu().numpy().view(np.uint64) == ov).all(), step
        now += 1000  # and so are these
        g.expire(now)
        o.expire(now)
    assert g.sync_status() == 0
