"""Large batches into L2-sized tables that are nearly full: find-or-put by sectors (128-bit keys: by halves) through
every bucket size, past the last of few hash functions into the stash and the overflow set, with values, with appended
keys, and with keys whose slots always read as free.  Batches of 2^19 keys and more take these kernels; every answer
is checked (exact)."""
import pytest
import torch

import paper_1712_09494_gb300 as ht
from workloads import device_keys as dk

pytestmark = pytest.mark.gpu

MANY = (1 << 19) + 17                                   # keys of a batch: sectors from 2^19 on, and a ragged tile


def _keys(n, kw, seed):
    idx = torch.arange(n, device="cuda")
    if kw == 32:
        x = dk.mix32_perm_dev(idx, seed)
        return (x - ((x >> 31) << 32)).to(torch.int32)
    return dk.mix63_perm_dev(idx, seed)


def _pick(lo, hi, size, seed):
    """`size` key numbers below hi, in random order: each of lo..hi once, twice or more often, and others below lo."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    new = torch.arange(lo, hi, device="cuda")
    rest = torch.randint(0, hi, (size - len(new),), device="cuda", generator=g)
    return torch.cat([new, rest])[torch.randperm(size, device="cuda", generator=g)]


def _new(pick, flags, n):
    return torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, pick, flags.to(torch.int64))


def _between(n, lo, hi):
    at = torch.arange(n, device="cuda")
    return ((at >= lo) & (at < hi)).to(torch.int64)


# Bucket slots, hash functions, and a load at which 300 to 1200 keys find all k buckets full: more than the stash's 101
# entries, fewer than the overflow set's 4096.
SHAPES = [(8, 1, 0.45), (16, 1, 0.6), (32, 1, 0.7), (8, 3, 0.8), (16, 3, 0.88), (32, 3, 0.93), (8, 16, 0.97), (16, 16, 0.98),
          (32, 16, 0.99)]


def _params(bs, k):
    return dict(bucket_slots=bs, lanes_per_key=4, num_hashes=k)


@pytest.mark.parametrize("kw", [32, 64])
@pytest.mark.parametrize("bs,k,load", SHAPES)
def test_sectors_of_a_nearly_full_table(kw, bs, k, load):
    slots = 1 << 18
    n = int(slots * load)
    keys = _keys(2 * n, kw, bs + k)
    t = ht.HashTable(slots, "bucket", kw, _params(bs, k))
    out = torch.empty_like(keys[:n])
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    stored = 0
    for i, upto in enumerate((n // 2, n - n // 8, n)):
        pick = _pick(stored, upto, MANY, i)
        flags = torch.full((MANY,), 7, dtype=torch.uint8, device="cuda")
        if i == 1:                                       # the new keys are appended, too
            ht.ht_find_or_put_append(t.handle, keys[pick], out, count, flags)
            assert int(count) == upto - stored
            assert torch.equal(torch.sort(out[:upto - stored])[0], torch.sort(keys[stored:upto])[0])
        else:
            ht.ht_find_or_put(t.handle, keys[pick], flags)
        assert torch.equal(_new(pick, flags, n), _between(n, stored, upto))
        stored = upto
    found, _ = t.lookup(keys)
    assert torch.equal(found, _between(2 * n, 0, n).to(torch.uint8))
    stats = ht.ht_stats(t.handle)
    assert stats["size"] == n and stats["dropped"] == 0
    assert stats["stash_used"] == 101 and stats["overflow_used"] > 0      # past the last bucket


@pytest.mark.parametrize("bs,k,load", SHAPES)
def test_sectors_of_a_nearly_full_map(bs, k, load):
    slots = 1 << 18
    n = int(slots * load)
    keys = _keys(2 * n, 32, bs + k)
    t = ht.HashTable(slots, "bucket", 32, _params(bs, k))
    value = (torch.arange(n, device="cuda") * 7 + 1).to(torch.int32)
    stored = 0
    for i, upto in enumerate((n // 2, n)):
        pick = _pick(stored, upto, MANY, i)
        t.insert(keys[pick], value[pick] + torch.where(pick < stored, 5, 0).to(torch.int32))   # stored keys keep theirs
        stored = upto
    found, v = t.lookup(keys)
    assert torch.equal(found, _between(2 * n, 0, n).to(torch.uint8))
    assert torch.equal(v[:n], value) and not bool(v[n:].any())
    assert ht.ht_stats(t.handle)["size"] == n and ht.ht_stats(t.handle)["dropped"] == 0


@pytest.mark.parametrize("ones", [False, True])
@pytest.mark.parametrize("k,load", [(1, 0.45), (3, 0.8), (16, 0.97)])
def test_halves_of_a_nearly_full_table_of_128_bit_keys(k, load, ones):
    """ones: every low word all ones, so that every stored key reads as a claim candidate."""
    slots = 1 << 18
    n = int(slots * load)
    high = _keys(2 * n, 64, k)
    low = torch.full_like(high, -1) if ones else _keys(2 * n, 64, k + 50)
    keys = torch.stack([low, high], dim=1).contiguous()
    t = ht.HashTable(slots, "bucket", 128, dict(num_hashes=k))
    out = torch.empty_like(keys[:n])
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    stored = 0
    for i, upto in enumerate((n // 2, n - n // 8, n)):
        pick = _pick(stored, upto, MANY, i)
        flags = torch.full((MANY,), 7, dtype=torch.uint8, device="cuda")
        if i == 1:
            ht.ht_find_or_put_append(t.handle, keys[pick], out, count, flags)
            assert int(count) == upto - stored
            assert torch.equal(torch.sort(out[:upto - stored, 1])[0], torch.sort(high[stored:upto])[0])
        else:
            ht.ht_find_or_put(t.handle, keys[pick], flags)
        assert torch.equal(_new(pick, flags, n), _between(n, stored, upto))
        stored = upto
    found, _ = t.lookup(keys)
    assert torch.equal(found, _between(2 * n, 0, n).to(torch.uint8))
    stats = ht.ht_stats(t.handle)
    assert stats["size"] == n and stats["dropped"] == 0
    assert stats["overflow_used"] > 0                    # past the last bucket
