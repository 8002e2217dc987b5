"""Small insert batches, with repeated keys, into tables that are nearly or wholly
full, where the wide searches run: at most 64 keys in one cluster, up to 2048 in a
cluster and a launch for what it leaves, more in the chain."""

import numpy as np
import pytest

from gpu_layout import download
from paper_1712_09624_gb300 import workload as W

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 33, 63, 64, 65, 255, 256, 257, 1000, 2048, 2049]


def fill_until(g, nb, share, now, ttl, seed):
    """Batches of new keys, a small share of the table each, until the share of the slots is taken."""
    pool, at, step = W.make_keys(seed, 75, 4 * nb * 8), int(0.9 * nb * 8), nb // 32
    g.insert(pool[:at], np.arange(at, dtype=np.uint64), now, ttl)
    while g.stats(now)["n_occupied"] < share * nb * 8:
        g.insert(pool[at:at + step], np.arange(at, at + step, dtype=np.uint64), now, ttl)
        at += step
        assert at + step <= pool.shape[0]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("share", [0.97, 0.99, 1.0])
@pytest.mark.parametrize("timers", [False, True])
def test_small_batches_into_full_tables(n, share, timers):
    from paper_1712_09624_gb300 import _ckpp as K
    from paper_1712_09624_gb300.table import FlowTable
    nb, now, ttl = 1 << 11, 7, 900 if timers else 0
    g = FlowTable(nb, timers=timers, seed=n)
    fill_until(g, nb, share, now, ttl, 800 + n)
    before = download(g).live(now)
    rng = np.random.default_rng(4000 + n)
    which = np.where(rng.random(n) < 0.2, rng.integers(0, n, n), np.arange(n))
    keys, vals = W.make_keys(900 + n, 76, n)[which], rng.integers(1, 2**62, n).astype(np.uint64)
    st = g.insert(keys, vals, now, ttl).cpu().numpy()
    first = np.array([np.flatnonzero(which == w)[0] for w in which])
    last = np.array([np.flatnonzero(which == w)[-1] for w in which])
    own = st[first]  # a group's first key reports the outcome, the others UPDATED or FULL as well
    assert set(own) <= {K.ST_INSERTED, K.ST_FULL}
    assert (st == np.where((first == np.arange(n)) | (own == K.ST_FULL), own, K.ST_UPDATED)).all()
    v, f = g.lookup(keys, now)
    stored = own == K.ST_INSERTED
    assert (f.cpu().numpy() == stored).all()
    assert (v.cpu().numpy().view(np.uint64) == np.where(stored, vals[last], 0)).all()
    d = download(g)
    assert d.check() == [] and len(d.live(now)) == len(before) + int((st == K.ST_INSERTED).sum())
    if len(before) == nb * 8:
        assert (st == K.ST_FULL).all()
    if n == 1 and share < 0.98:
        assert st[0] == K.ST_INSERTED
    assert g.sync_status() == 0
