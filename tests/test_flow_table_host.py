"""What FlowTable decides on the host, before a kernel is launched."""

import numpy as np
import pytest
import torch

from paper_1712_09624_gb300 import _ckpp as K
from paper_1712_09624_gb300.table import FlowTable


@pytest.fixture
def table():
    t = FlowTable.__new__(FlowTable)  # no device buffer, no handle: host buffers stand in
    t.device, t.handle, t._ws = torch.device("cpu"), None, None
    return t


@pytest.mark.parametrize("n,values", [(1, 0), (5, 4), (3, 3), (3, 7)])
@pytest.mark.parametrize("as_array", [False, True])
def test_insert_refuses_fewer_values_than_keys(table, monkeypatch, n, values, as_array):
    calls = []
    monkeypatch.setattr(K, "table_insert", lambda handle, k, v, *rest: calls.append((k.shape[0], v.numel())))
    k, v = np.zeros((n, 16), np.uint8), np.zeros(values, np.int64)
    if not as_array:
        k, v = torch.from_numpy(k), torch.from_numpy(v)
    if values < n:
        with pytest.raises(ValueError):
            table.insert(k, v)
        assert calls == []
    else:
        assert table.insert(k, v).shape == (n,) and calls == [(n, values)]


@pytest.mark.parametrize("first", [0, 100, (1 << 30) + 1])
def test_workspace_suits_every_batch_after_one_that_is_too_large(table, first):
    table.workspace(first)
    table.workspace((1 << 30) + 1)
    for n in (1, 99, 5000, 200):
        assert table.workspace(n).numel() >= K.ckpp_workspace_bytes(n) > 0, n
