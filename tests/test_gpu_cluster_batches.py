"""Small write batches (one launch of one cluster) into a crowded table, so that
the lanes of a warp reach the barriers between its stages by different ways: keys
that find a slot at once, keys that wait for locks along a cuckoo path, repeated
keys and keys beyond the end of the batch."""

import numpy as np
import pytest

import oracle
from gpu_layout import download, oracle_live
from paper_1712_09624_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [255, 256, 257, 700, 1031, 2048])
@pytest.mark.parametrize("timers", [False, True])
def test_crowded_cluster_batches_match_the_oracle(n, timers):
    from paper_1712_09624_gb300.table import FlowTable
    nb, now, ttl = n, 20, 900
    rng = np.random.default_rng(3000 + n)
    g, o = FlowTable(nb, timers=timers, seed=n), oracle.Table(nb, 8, timers, n)
    f = W.fill(600 + n, int(0.83 * nb * 8))
    t = ttl if timers else 0
    assert (g.insert(f.keys, f.values, now, t).cpu().numpy() == o.insert(f.keys, f.values, now, t)).all()
    fresh = W.make_keys(700 + n, 74, n)
    for step in range(4):  # to a load of 0.93 and back
        keys = fresh[np.where(rng.random(n) < 0.2, rng.integers(0, n, n), np.arange(n))]
        vals = rng.integers(0, 2**62, n).astype(np.uint64)
        assert (g.insert(keys, vals, now, t).cpu().numpy() == o.insert(keys, vals, now, t)).all(), step
        d = download(g)
        assert d.check() == [] and d.live(now) == oracle_live(o, now), step
        keys = keys[rng.permutation(n)]
        assert (g.delete(keys, now).cpu().numpy() == o.delete(keys, now)).all(), step
        d = download(g)
        assert d.check() == [] and d.live(now) == oracle_live(o, now), step
    assert g.sync_status() == 0
