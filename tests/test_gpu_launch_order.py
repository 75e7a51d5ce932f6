"""Kernels that start early (programmatic stream serialisation) must still see
all writes of the ones before them: chains of small calls without a
synchronisation, mixed with torch kernels, on a side stream, and captured into
a CUDA graph and replayed."""
import numpy as np
import pytest
import torch

import paper_1712_09494_gb300 as ht
from workloads import device_keys as dk

pytestmark = pytest.mark.gpu


def _keys(n, width, seed):
    k = dk.distinct_keys_dev(n, seed, device="cuda")
    if width == 32:
        m = dk.mix32_perm_dev(torch.arange(n, device="cuda"), seed)
        return (m - ((m >> 31) << 32)).to(torch.int32)
    return k if width == 64 else torch.stack([dk.mix63_perm_dev(k, seed + j) for j in range(width // 64)], dim=1).contiguous()


@pytest.mark.parametrize("scheme", ["bucket", "cuckoo"])
@pytest.mark.parametrize("width", [32, 64, 128, 256])
def test_chains_of_small_calls(scheme, width):
    n = 3000
    keys = _keys(2 * n, width, 5)
    t = ht.HashTable(int(n / 0.8), scheme, width)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    with torch.cuda.stream(side):
        for r in range(200):
            t.clear()
            a = t.find_or_put(keys[:n // 2])
            b = t.find_or_put(keys[:n])             # half of them just stored
            # Keys that a torch kernel has just written.
            moved = keys.roll(1, 0)
            found, _ = t.lookup(moved)
            want = torch.zeros(2 * n, dtype=torch.uint8, device="cuda")
            want[1:n + 1] = 1
            bad += (a != 1).sum() + b[:n // 2].sum() + (b[n // 2:] != 1).sum() + (found != want).sum()
    side.synchronize()
    assert int(bad) == 0 and t.sync(side) == 0 and t.size(side) == n


@pytest.mark.parametrize("scheme", ["bucket", "cuckoo"])
@pytest.mark.parametrize("slots,n", [(4000, 3000), (24_000_000, 3_000_000)])
def test_captured_and_replayed(scheme, slots, n):
    """Also a batch that would be reordered: its scratch may not be made during a capture."""
    keys = _keys(n, 64, 9)
    t = ht.HashTable(slots, scheme, 64)
    flags = torch.empty(n, dtype=torch.uint8, device="cuda")
    found = torch.empty(n, dtype=torch.uint8, device="cuda")

    def calls():
        ht.ht_clear(t.handle)
        ht.ht_find_or_put(t.handle, keys, flags)
        ht.ht_lookup(t.handle, keys, None, found)

    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        calls()
    for r in range(3):
        flags.zero_()
        found.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert bool(flags.all()) and bool(found.all())
    calls()                                          # and not captured, with the scratch
    assert t.size() == n and bool(flags.all())
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2):
        calls()
    flags.zero_()
    g2.replay()
    torch.cuda.synchronize()
    assert bool(flags.all()) and t.size() == n


def test_a_failed_allocation_is_no_later_calls_error():
    keys = _keys(1000, 64, 1)
    small = ht.HashTable(4000, "bucket", 64)
    flags = torch.empty(1000, dtype=torch.uint8, device="cuda")
    out = torch.empty(1000, dtype=torch.int64, device="cuda")
    for r in range(2):
        for scheme in ("bucket", "cuckoo"):
            with pytest.raises(ht.HtError) as err:
                ht.HashTable(1 << 39, scheme, 64)            # 4 TB
            assert err.value.status == 2
            small.clear()
            ht.ht_multi_find_or_put([small.handle], [(0, keys, flags)])
            count = torch.zeros(1, dtype=torch.int64, device="cuda")
            ht.ht_compact(keys, flags, out, count)
            assert int(count) == 1000 and small.size() == 1000
