"""The two forms of the plain lookup (one thread per key for tables that stay in
L2, whole bucket lines for larger ones) against known answers and each other, at
the batch sizes of warps and blocks and at table sizes on both sides of the line
between them. Host buffers and refreshing lookups always take the second form."""

import numpy as np
import pytest
import torch

from paper_1712_09624_gb300 import workload as W

pytestmark = pytest.mark.gpu


def pinned(a):
    t = torch.empty(a.shape, dtype=a.dtype, pin_memory=True)
    t.copy_(a)
    return t


@pytest.mark.parametrize("nb", [2, 777, 1 << 20, (1 << 20) + 1])
@pytest.mark.parametrize("timers", [False, True])
def test_lookup_forms_agree(nb, timers):
    from paper_1712_09624_gb300 import _ckpp as K
    from paper_1712_09624_gb300.table import FlowTable
    m = min(int(0.8 * nb * 8), 300_000)
    f = W.fill(500 + nb, m)
    g = FlowTable(nb, timers=timers, seed=nb)
    dead = m // 3 if timers else 0
    if dead:  # the first third is dead at the time of the lookups
        assert (g.insert(f.keys[:dead], f.values[:dead], 10, 5).cpu().numpy() == K.ST_INSERTED).all()
    assert (g.insert(f.keys[dead:], f.values[dead:], 10, 900).cpu().numpy() == K.ST_INSERTED).all()
    now = 30
    for n in (1, 31, 33, 255, 256, 257, 100_003):
        q = W.lookup_batch(nb, n, f, 0.4, batch_id=n)
        want = q.expect_found.astype(bool) & (~q.expect_found.astype(bool) | (q.expect_value >= dead))
        vals = np.where(want, q.expect_value, 0).astype(np.uint64)
        v, fd = g.lookup(q.keys, now)
        assert (fd.cpu().numpy() == want).all() and (v.cpu().numpy().view(np.uint64) == vals).all(), n
        hk = pinned(torch.from_numpy(q.keys))
        hv, hf = torch.empty(n, dtype=torch.int64, pin_memory=True), torch.empty(n, dtype=torch.bool, pin_memory=True)
        K.ckpp_bulk_lookup(g.handle, hk, hv, hf, now)
        torch.cuda.synchronize()
        assert torch.equal(hv, v.cpu()) and torch.equal(hf, fd.cpu()), n
        if timers:
            rv, rf = g.lookup(q.keys, now, 900)
            assert torch.equal(rv, v) and torch.equal(rf, fd), n
            again = g.lookup(q.keys, now + 899)[1]  # refreshed hits outlive their first time to live
            assert torch.equal(again, fd), n
