"""Device pointers that are aligned to their words but not to the wider accesses
that kernels make: accepted ones give the same results, others are refused on
the host."""
import numpy as np
import pytest
import torch

import paper_1712_09494_gb300 as ht
from gpu_util import assert_same_set, to_dev, to_np
from workloads import keys as wk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("nslots", [1, 2, 1000, 75_001])
def test_noalloc_table_at_any_word(offset, nslots):
    """The caller's table carved out of an arena at an even or an odd word: emptied from its first to its last word,
    and none beside it."""
    arena = torch.full((nslots + 4,), 77, dtype=torch.int64, device="cuda")
    slots = arena[1 + offset:1 + offset + nslots]
    assert slots.data_ptr() % 16 == 8 * (1 - offset)
    state = torch.empty(ht.NOALLOC_STATE_BYTES, dtype=torch.uint8, device="cuda")
    n = max(1, int(nslots * 0.6))
    keys = wk.distinct_keys(n, 64, seed=nslots)
    got = torch.empty(n, dtype=torch.uint8, device="cuda")
    ht.ht_cuckoo_find_or_put_noalloc(slots, state, 5, to_dev(keys), got, reset=True)
    torch.cuda.synchronize()
    assert to_np(got).all()
    words = to_np(slots.clone(), np.uint64)
    spilled = to_np(state[128:1152 + 512].clone(), np.uint64)
    held = np.concatenate([words, spilled])
    assert_same_set(held[held != np.uint64(2 ** 64 - 1)], keys)
    assert (to_np(arena[:1 + offset]) == 77).all() and (to_np(arena[1 + offset + nslots:]) == 77).all()
