"""Each call takes its place in stream order, eagerly and in a captured graph:
kernels and copies queued right before it write its keys and values in place,
on its own stream and on one that joins it, and the same buffers are written
anew right after it."""

import numpy as np
import pytest
import torch

import oracle
from gpu_layout import download, oracle_live
from paper_1712_09624_gb300 import workload as W

pytestmark = pytest.mark.gpu

ROUNDS = 4


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("n,nb", [(50, 500), (300, 500), (2048, 4000), (5000, (1 << 20) + 1), (70001, 30000)])
def test_calls_follow_what_was_queued_before_them(n, nb, captured):
    from paper_1712_09624_gb300 import _ckpp as K
    from paper_1712_09624_gb300.batched import BatchedLookup
    from paper_1712_09624_gb300.table import FlowTable
    g, o = FlowTable(nb, seed=n), oracle.Table(nb, 8, False, n)
    batch = BatchedLookup([g], max_jobs=1)
    pool = W.make_keys(500 + n, 73, 2 * n)
    base = torch.from_numpy(pool).cuda()
    pick = torch.empty((3, n), dtype=torch.int64, device="cuda")  # the keys of the insert, the lookups, the delete
    keys = torch.zeros((n, 16), dtype=torch.uint8, device="cuda")
    staged, vals = (torch.zeros(n, dtype=torch.int64, device="cuda") for _ in range(2))
    inserted, deleted = (torch.empty(n, dtype=torch.uint8, device="cuda") for _ in range(2))
    v1, v2 = (torch.empty(n, dtype=torch.int64, device="cuda") for _ in range(2))
    f1, f2 = (torch.empty(n, dtype=torch.bool, device="cuda") for _ in range(2))
    ws = torch.empty(K.ckpp_workspace_bytes(n), dtype=torch.uint8, device="cuda")
    load = torch.zeros(1 << 24, device="cuda")  # keeps the stream busy while the rest is queued
    batch.set_jobs([(0, keys, v2, f2)])
    side = torch.cuda.Stream()

    def calls():
        for _ in range(3):
            load.add_(1.0)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            vals.copy_(staged)
        torch.index_select(base, 0, pick[0], out=keys)
        torch.cuda.current_stream().wait_stream(side)
        K.ckpp_bulk_insert(g.handle, keys, vals, inserted, ws)
        torch.index_select(base, 0, pick[1], out=keys)
        K.ckpp_bulk_lookup(g.handle, keys, v1, f1)
        batch.launch()
        keys.zero_()  # a memset right before and a copy right after a kernel
        torch.index_select(base, 0, pick[2], out=keys)
        K.ckpp_bulk_delete(g.handle, keys, deleted, ws)
        keys.zero_()
        vals.zero_()

    rng = np.random.default_rng(n)
    s = torch.cuda.Stream()
    graph = None
    for step in range(ROUNDS):
        p = rng.integers(0, 2 * n, (3, n))
        v = rng.integers(0, 2**62, n)
        torch.cuda.synchronize()
        pick.copy_(torch.from_numpy(p))
        staged.copy_(torch.from_numpy(v))
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            if captured and step == 1:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=s):
                    calls()
            if graph is not None:
                graph.replay()
            else:
                calls()
        torch.cuda.synchronize()
        assert (inserted.cpu().numpy() == o.insert(pool[p[0]], v.astype(np.uint64))).all(), step
        ov, of = o.lookup(pool[p[1]])
        for gv, gf in ((v1, f1), (v2, f2)):
            assert (gf.cpu().numpy() == of).all() and (gv.cpu().numpy().view(np.uint64) == ov).all(), step
        assert (deleted.cpu().numpy() == o.delete(pool[p[2]])).all(), step
        d = download(g)
        assert d.check() == [] and d.live(0) == oracle_live(o, 0), step
