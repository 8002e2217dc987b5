"""Insert and delete batches of one shard's keys, as each rank of a sharded table
gets them from the partition: they share bits 16-31 of the primary hash. Against
the oracle, at the sizes of the cluster form, its edge and large batches."""

import numpy as np
import pytest
import torch

import oracle
from gpu_layout import download, oracle_live

pytestmark = pytest.mark.gpu


def shard_keys(n, n_shards, seed):
    """n keys of the first shard, as ckpp_shard_partition finds them."""
    from paper_1712_09624_gb300 import _ckpp as K
    total = n * n_shards + 8 * int((n * n_shards) ** 0.5) * n_shards
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    keys = torch.randint(-(2**63), 2**63 - 1, (total, 2), generator=g, device="cuda").view(torch.uint8).view(total, 16)
    pos, ks = torch.empty(total, dtype=torch.int32, device="cuda"), torch.empty_like(keys)
    counts = torch.empty(n_shards, dtype=torch.int64, device="cuda")
    ws = torch.empty(K.ckpp_shard_workspace_bytes(total, n_shards), dtype=torch.uint8, device="cuda")
    K.ckpp_shard_partition(keys, None, seed, n_shards, pos, ks, None, counts, ws)
    assert int(counts[0]) >= n
    return ks[:n].cpu().numpy()


@pytest.mark.parametrize("n,n_shards", [(2048, 64), (2049, 64), (32768, 8), (32768, 64), (1 << 20, 1), (1 << 20, 8),
                                        (1 << 18, 64)])
def test_batches_of_one_shard_match_the_oracle(n, n_shards):
    from paper_1712_09624_gb300.table import FlowTable
    seed, nb = 31, n // 4
    g, o = FlowTable(nb, seed=seed), oracle.Table(nb, 8, False, seed)
    rng = np.random.default_rng(n + n_shards)
    own = shard_keys(n, n_shards, seed)
    for step in range(2):
        keys = own[np.where(rng.random(n) < 0.05, rng.integers(0, n, n), rng.permutation(n))]
        vals = rng.integers(0, 2**62, n).astype(np.uint64)
        assert (g.insert(keys, vals).cpu().numpy() == o.insert(keys, vals)).all(), step
        keys = keys[rng.random(n) < 0.5]
        assert (g.delete(keys).cpu().numpy() == o.delete(keys)).all(), step
        v, f = g.lookup(own)
        ov, of = o.lookup(own)
        assert (f.cpu().numpy() == of).all() and (v.cpu().numpy().view(np.uint64) == ov).all(), step
    d = download(g)
    assert d.check() == [] and d.live(0) == oracle_live(o, 0)
