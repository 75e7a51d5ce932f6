"""Bucket tables almost full: most keys find their first buckets full and go
through the kernels' queues of unsettled keys, past the last bucket into the
stash and the overflow set, at batch sizes around the 32-key tile and the
queue's limits.  Every answer must equal the oracle's (exact)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1712_09494_gb300 as ht
from gpu_util import assert_flags_per_key, assert_same_set, to_dev, to_np
from workloads import keys as wk

pytestmark = pytest.mark.gpu

SHAPES = [(8, 2), (8, 8), (16, 2), (16, 4), (16, 16), (32, 4), (32, 32)]


def _batches(keys, rng):
    """Ragged batches over the keys, each with a third of repeats (also inside the batch)."""
    out, at = [], 0
    sizes = [1, 31, 32, 33, 63, 64, 65, 257]
    i = 0
    while at < len(keys):
        m = min(sizes[i % len(sizes)], len(keys) - at)
        fresh = keys[at:at + m]
        rep = keys[rng.integers(0, at + m, size=m // 3)]
        out.append(rng.permutation(np.concatenate([fresh, rep])))
        at += m
        i += 1
    return out


@pytest.mark.parametrize("kw", [32, 64])
@pytest.mark.parametrize("bs,lanes", SHAPES)
@pytest.mark.parametrize("k", [1, 3, 16])
def test_nearly_full_table_settles_every_key(kw, bs, lanes, k):
    slots = 2048
    n = int(slots * (1.02 if k == 1 else 0.98))        # k = 1: past the table into the spill
    keys = wk.distinct_keys(n, kw, seed=bs * 100 + lanes + k)
    rng = np.random.default_rng(k)
    t = ht.HashTable(slots, "bucket", kw, dict(bucket_slots=bs, lanes_per_key=lanes, num_hashes=k, max_rebuilds=1))
    orc = oracle.OracleTable()
    batches = _batches(keys, rng)
    batches.append(rng.permutation(np.concatenate([keys, keys])))      # one large batch of repeats
    for b in batches:
        assert_flags_per_key(b, to_np(t.find_or_put(to_dev(b))), orc.find_or_put(b))
    q = np.concatenate([keys, wk.distinct_keys(n, kw, seed=bs * 100 + lanes + k, start=n)])
    found, _ = t.lookup(to_dev(q))
    assert np.array_equal(to_np(found), np.repeat(np.array([1, 0], dtype=np.uint8), n))
    got, _ = t.export()
    assert_same_set(to_np(got, np.uint32 if kw == 32 else np.uint64), keys)


def test_values_of_queued_keys():
    n = 2000
    keys = wk.distinct_keys(n, 32, seed=4)
    t = ht.HashTable(2048, "bucket", 32)
    vals = np.arange(n, dtype=np.uint32) * 7 + 1
    t.insert(to_dev(keys), to_dev(vals))
    found, v = t.lookup(to_dev(keys))
    assert to_np(found).all() and np.array_equal(to_np(v, np.uint32), vals)


def test_many_nearly_full_tables_in_one_call():
    n, tables = 250, 40                                # 256-slot tables
    tabs = [ht.HashTable(256, "bucket", 64) for _ in range(tables)]
    keys = [wk.distinct_keys(n, 64, seed=50 + i) for i in range(tables)]
    for lo, hi in ((0, 100), (50, n)):
        items, flags = [], []
        for i in range(tables):
            flags.append(torch.zeros(hi - lo, dtype=torch.uint8, device="cuda"))
            items.append((i, to_dev(keys[i][lo:hi]), flags[-1]))
        ht.ht_multi_find_or_put([t.handle for t in tabs], items)
        for i in range(tables):
            new = np.arange(lo, hi) >= (0 if lo == 0 else 100)
            assert np.array_equal(to_np(flags[i]), new.astype(np.uint8))
    assert [t.size() for t in tabs] == [n] * tables


@pytest.mark.parametrize("lanes", [2, 4])
@pytest.mark.parametrize("ones", [False, True])
def test_nearly_full_table_of_128_bit_keys(lanes, ones):
    """ones: every low word all ones, so that every stored key reads as a claim candidate."""
    n = 1000
    hi = wk.distinct_keys(2 * n, 64, seed=lanes)
    lo = np.full(2 * n, 2 ** 64 - 1, dtype=np.uint64) if ones else wk.distinct_keys(2 * n, 64, seed=9)
    keys = np.stack([lo, hi], axis=1)
    rng = np.random.default_rng(lanes)
    t = ht.HashTable(1024, "bucket", 128, dict(bucket_slots=8, lanes_per_key=lanes))
    orc = oracle.OracleTable128()
    for idx in _batches(np.arange(n), rng) + [rng.permutation(np.tile(np.arange(n), 2))]:
        got = to_np(t.find_or_put(to_dev(keys[idx])))
        assert_flags_per_key(idx, got, orc.find_or_put(keys[idx]))
    found, _ = t.lookup(to_dev(keys))
    assert np.array_equal(to_np(found), np.repeat(np.array([1, 0], dtype=np.uint8), n))
    assert t.sync() == 0 and t.size() == n


@pytest.mark.parametrize("bs,lanes", [(8, 2), (16, 2), (32, 4)])
@pytest.mark.parametrize("kw", [32, 64])
def test_table_past_l2_at_high_load(kw, bs, lanes):
    """Tables larger than L2 (other kernels than small ones) at load 0.95: every batch's fresh keys are new and its
    repeats are not, all stored keys are found with their values and no other key is."""
    from workloads import device_keys as dk
    slots = 24_000_000                                  # 192 MB
    n = int(slots * 0.95)
    idx = torch.arange(2 * n, dtype=torch.int64, device="cuda")
    if kw == 64:
        keys = dk.mix63_perm_dev(idx, bs)
    else:
        k = dk.mix32_perm_dev(idx, bs)
        keys = (k - ((k >> 31) << 32)).to(torch.int32)
    t = ht.HashTable(slots, "bucket", kw, dict(bucket_slots=bs, lanes_per_key=lanes))
    vals = (idx[:n] * 3 + 1).to(torch.int32)
    at = 0
    for m in (n // 2 + 7, n // 4 + 13, 1, 31, n):
        m = min(m, n - at)
        rep = torch.randint(0, at, (m // 4,), device="cuda") if at else idx[:0]
        if at == 0 and kw == 32:
            t.insert(keys[:m], vals[:m])                # the rest of the keys get value 0
        else:
            order = torch.randperm(m + len(rep), device="cuda")
            batch = torch.cat([keys[at:at + m], keys[rep]])[order]
            assert torch.equal(t.find_or_put(batch), (order < m).to(torch.uint8))
        if at == 0:
            first = m
        at += m
    found, v = t.lookup(keys)
    assert torch.equal(found, (idx < n).to(torch.uint8))
    if kw == 32:
        want = torch.zeros(2 * n, dtype=torch.int32, device="cuda")
        want[:first] = vals[:first]
        assert torch.equal(v, want)
    assert t.sync() == 0 and t.size() == n


@pytest.mark.parametrize("w", [3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("digest_bits", [0, 6])
def test_nearly_full_table_of_long_keys(w, digest_bits):
    """Rows of every word count; few digest bits make most matching tags another key's."""
    n = 960
    keys = wk.distinct_keys(2 * n, 64 * w, seed=w, shared_prefix=True)
    rng = np.random.default_rng(w)
    t = ht.HashTable(1024 if not digest_bits else 4096, "bucket", 64 * w, dict(digest_bits=digest_bits))
    orc = oracle.OracleTableLong(w)
    for idx in _batches(np.arange(n), rng) + [rng.permutation(np.tile(np.arange(n), 2))]:
        got = to_np(t.find_or_put(to_dev(keys[idx])))
        assert_flags_per_key(idx, got, orc.find_or_put(keys[idx]))
    found, _ = t.lookup(to_dev(keys))
    assert np.array_equal(to_np(found), np.repeat(np.array([1, 0], dtype=np.uint8), n))
    assert t.sync() == 0 and t.size() == n
    got, _ = t.export()
    assert set(map(tuple, to_np(got, np.uint64).tolist())) == set(map(tuple, keys[:n].tolist()))


@pytest.mark.parametrize("scheme,kw", [("bucket", 32), ("bucket", 64), ("bucket", 128), ("cuckoo", 32), ("cuckoo", 64)])
def test_large_batches_are_reordered_by_table_region(scheme, kw):
    """Batches with more keys than the table (past L2) has lines, taken region by region: whole pieces of 2^24 keys
    with a ragged one after them, batches with and without flags, appended keys, repeats in other batches, and an
    odd flag address."""
    from workloads import device_keys as dk
    slots = 24_000_000                                  # 192 MB: 1.5 M lines
    n = int(slots * 0.85)
    idx = torch.arange(2 * n, dtype=torch.int64, device="cuda")
    if kw >= 64:
        keys = dk.mix63_perm_dev(idx, 3)
    else:
        k = dk.mix32_perm_dev(idx, 3)
        keys = (k - ((k >> 31) << 32)).to(torch.int32)
    if kw == 128:                                       # low words of all ones among them
        keys = torch.stack([torch.where(idx % 5 == 0, torch.full_like(keys, -1), keys), keys], dim=1).contiguous()
    t = ht.HashTable(slots, scheme, kw)
    order = torch.randperm(n, device="cuda")
    first = keys[:n][order][:2_000_001]                 # a ragged tile
    flags = torch.full((len(first) + 8,), 7, dtype=torch.uint8, device="cuda")
    ht.ht_find_or_put(t.handle, first, flags[3:3 + len(first)])
    assert bool((flags[3:3 + len(first)] == 1).all()) and flags[:3].tolist() == [7] * 3
    assert flags[3 + len(first):].tolist() == [7] * 5
    t.insert(keys[:n][order][1_000_000:5_000_000])      # no flags
    every = torch.randperm(n, device="cuda")            # n > 2^24: a whole piece and the rest
    new = torch.empty(n, dtype=torch.uint8, device="cuda")
    out = torch.empty_like(keys[:n])
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    ht.ht_find_or_put_append(t.handle, keys[:n][every], out, count, new)
    stored = torch.zeros(n, dtype=torch.bool, device="cuda")
    stored[order[:5_000_000]] = True
    assert torch.equal(new, (~stored[every]).to(torch.uint8))
    assert int(count) == n - 5_000_000
    own = (lambda x: x[:, 1]) if kw == 128 else (lambda x: x)       # the word that tells keys apart
    assert torch.equal(torch.sort(own(out[:int(count)]))[0], torch.sort(own(keys[:n][~stored]))[0])
    found, _ = t.lookup(keys)
    assert torch.equal(found, (idx < n).to(torch.uint8))
    assert t.sync() == 0 and t.size() == n


def test_reordered_batch_of_one_key_and_reserved_keys():
    """Every key in one region, and reserved keys among them: skipped and reported."""
    t = ht.HashTable(24_000_000, "bucket", 64)
    keys = torch.full((3_000_000,), 12345, dtype=torch.int64, device="cuda")
    keys[1_000_000:] = torch.arange(2_000_000, device="cuda") + (1 << 40)
    keys[::1000] = -1
    flags = t.find_or_put(keys)
    assert int(flags[:1_000_000].sum()) == 1 and int(flags.sum()) == 1 + 2_000_000 - 2000
    assert int(flags[::1000].sum()) == 0
    assert t.sync() == 1 and t.size() == 1 + 2_000_000 - 2000


@pytest.mark.parametrize("k,h1,load,slots", [(2, 0, 0.4, 24_000_000), (4, 0, 0.85, 24_000_000), (4, 1, 0.85, 24_000_000),
                                             (8, 0, 0.9, 24_000_000), (4, 0, 0.1, 80_000_000)])
@pytest.mark.parametrize("kw", [32, 64])
def test_cuckoo_table_past_l2_in_the_batchs_order(kw, k, h1, load, slots):
    """Cuckoo tables larger than L2 with batches too small to be reordered: each key of a batch is new in exactly one
    of its two places, stored keys are not, and lookups return the stored values."""
    from workloads import device_keys as dk
    n = int(slots * load)                               # 192 and 640 MB; reordered from 1.9 and 6.3 M keys
    idx = torch.arange(2 * n, dtype=torch.int64, device="cuda")
    if kw == 64:
        keys = dk.mix63_perm_dev(idx, k)
    else:
        d = dk.mix32_perm_dev(idx, k)
        keys = (d - ((d >> 31) << 32)).to(torch.int32)
    t = ht.HashTable(slots, "cuckoo", kw, dict(num_hashes=k, cuckoo_chain_h1=h1))
    vals = (idx[:n] * 3 + 1).to(torch.int32)
    at = first = 0
    if kw == 32:
        at = first = n // 2 + 7
        t.insert(keys[:at], vals[:at])                  # the rest of the keys get value 0
    sizes = [1, 31, 33, 700_001]
    while at < n:
        m = min(sizes.pop(0) if sizes else 650_000, n - at)
        rep = torch.randint(0, at, (m // 2,), device="cuda") if at else idx[:0]
        order = torch.randperm(2 * m + len(rep), device="cuda")
        f = t.find_or_put(torch.cat([keys[at:at + m], keys[at:at + m], keys[rep]])[order])
        g = torch.zeros_like(f)
        g[order] = f
        assert bool((g[:m] + g[m:2 * m] == 1).all()) and not bool(g[2 * m:].any())
        at += m
    found, v = t.lookup(keys)
    assert torch.equal(found, (idx < n).to(torch.uint8))
    if kw == 32:
        want = torch.zeros(2 * n, dtype=torch.int32, device="cuda")
        want[:first] = vals[:first]
        assert torch.equal(v, want)
    assert t.sync() == 0 and t.size() == n
