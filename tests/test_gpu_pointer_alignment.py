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


def _rows(n, off):
    """An (n, 2) tensor whose first row is `off` words past a 16-byte boundary."""
    r = torch.zeros(2 * n + 1, dtype=torch.int64, device="cuda")[off:off + 2 * n].view(n, 2)
    assert r.is_contiguous() and r.data_ptr() % 16 == 8 * off
    return r


@pytest.mark.parametrize("scheme", ["bucket", "cuckoo"])
def test_128_bit_keys_off_a_16_byte_boundary_are_refused(scheme):
    n = 100
    t = ht.HashTable(256, scheme, 128)
    off, even = _rows(n, 1), _rows(n, 0)
    even[:, 0] = off[:, 0] = torch.arange(n, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    flags = torch.zeros(n, dtype=torch.uint8, device="cuda")
    calls = [lambda: t.find_or_put(off), lambda: t.insert(off), lambda: t.lookup(off),
             lambda: ht.ht_find_or_put_append(t.handle, off, even.clone(), count, flags),
             lambda: ht.ht_find_or_put_append(t.handle, even, _rows(n, 1), count, flags)]
    for call in calls:
        with pytest.raises(ht.HtError) as err:
            call()
        assert err.value.status == 1
    assert t.sync() == 0 and t.size() == 0 and int(count) == 0
    # No keys: no address to refuse; and the next calls work.
    ht.ht_find_or_put(t.handle, off[:0], None)
    assert bool(t.find_or_put(even).all()) and bool(t.lookup(off.clone())[0].all()) and t.size() == n


@pytest.mark.parametrize("scheme", ["bucket", "cuckoo"])
def test_128_bit_states_off_a_16_byte_boundary_are_refused(scheme):
    c, w = 16, 2                                           # 80 bits, two local states each
    deg = np.zeros((16, 32), dtype=np.uint8)
    tgt = np.zeros((16, 32, 4), dtype=np.uint8)
    deg[:, :w] = 1
    tgt[:, 0, 0] = 1
    model = ht.make_model(c, np.full(c, 5, dtype=np.uint8), deg, tgt, np.zeros((16, 32, 4), dtype=np.uint8),
                          np.zeros((0, 2), dtype=np.int64))
    n = w ** c
    t = ht.HashTable(2 * n, scheme, 128)
    with pytest.raises(ht.HtError) as err:
        ht.ht_bfs(t.handle, model, 0, 64, _rows(n, 1))
    assert err.value.status == 1
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    for states, succ in ((_rows(4, 1), _rows(64, 0)), (_rows(4, 0), _rows(64, 1))):
        with pytest.raises(ht.HtError) as err:
            ht.ht_successors(model, states, succ, count)
        assert err.value.status == 1
    assert int(count) == 0 and t.size() == 0
    states = _rows(n, 0)
    assert ht.ht_bfs(t.handle, model, 0, 64, states)[0].states == n
