"""Device memory of an exploration: the states it keeps for itself, where they are large, are free again when it
returns, without a synchronisation by the caller, whether it ends, is stopped or cannot be run."""
import math

import numpy as np
import pytest
import torch

import paper_1712_09494_gb300 as ht

pytestmark = pytest.mark.gpu

GB = 1 << 30


def _model(windows):
    c = len(windows)
    deg = np.zeros((16, 32), dtype=np.uint8)
    tgt = np.zeros((16, 32, 4), dtype=np.uint8)
    deg[:, :] = 1
    for i, w in enumerate(windows):
        tgt[i, :w, 0] = (np.arange(w) + 1) % w
    return ht.make_model(c, np.full(c, 5, dtype=np.uint8), deg, tgt, np.zeros((16, 32, 4), dtype=np.uint8),
                         np.zeros((0, 2), dtype=np.int64))


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("max_levels", [4096, 5])
def test_work_memory_is_free_on_return(fused, max_levels):
    windows = [5] * 9
    n = math.prod(windows)                                 # 2 M states
    t = ht.HashTable(2 * n, "bucket", 64)
    model = _model(windows)
    ht.ht_bfs(t.handle, model, 0, max_levels, None, states_cap=2 * n, fused=fused)      # what the table keeps
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    t.clear()
    res, _ = ht.ht_bfs(t.handle, model, 0, max_levels, None, states_cap=1 << 29, fused=fused)   # 4 GB of states
    after = torch.cuda.mem_get_info()[0]
    assert res.complete == (max_levels == 4096) and (res.states == n) == bool(res.complete)
    assert before - after < GB


def test_memory_of_an_exploration_that_cannot_be_had():
    t = ht.HashTable(1 << 20, "bucket", 64)
    model = _model([3] * 4)
    ht.ht_bfs(t.handle, model)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    t.clear()
    with pytest.raises(ht.HtError) as err:
        ht.ht_bfs(t.handle, model, 0, 4096, None, states_cap=1 << 39)                   # 4 TB
    assert err.value.status == 2
    assert before - torch.cuda.mem_get_info()[0] < GB
    assert ht.ht_bfs(t.handle, model)[0].states == 81
