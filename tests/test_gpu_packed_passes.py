"""Many tables in one call, by both passes of the packed kernel: buckets a sector at a time in launches of 2^19 keys
and more, whole below.  Tables nearly full, repeats inside the items and of earlier calls, both kinds of launch in turn
on the same tables."""
import pytest
import torch

import paper_1712_09494_gb300 as ht
from workloads import device_keys as dk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [32, 64])
@pytest.mark.parametrize("bs,k", [(8, 16), (16, 16), (16, 2), (32, 16)])
def test_few_and_many_keys_in_a_call(kw, bs, k):
    count, slots = 32, 20_000
    n = int(slots * (0.75 if k == 2 else 0.9))             # keys of each table at the end
    lanes = dict(bucket_slots=bs, lanes_per_key=4, num_hashes=k)
    tabs = [ht.HashTable(slots, "bucket", kw, lanes) for _ in range(count)]
    base = torch.arange(count * n, device="cuda").view(count, n)
    keys = dk.mix63_perm_dev(base.flatten(), bs).view(count, n)
    if kw == 32:
        x = dk.mix32_perm_dev(base.flatten(), bs).view(count, n)
        keys = (x - ((x >> 31) << 32)).to(torch.int32)
    stored = 0
    g = torch.Generator(device="cuda")
    g.manual_seed(bs)
    # Few keys (8 or 300 a table), many (16400 and more a table: 2^19 in all), few, many, the rest.
    for upto, size in ((5, 8), (n // 2, 16_400), (n // 2 + 100, 300), (n - 60, 16_700), (n, 100)):
        pick = torch.randint(0, upto, (count, size), device="cuda", generator=g)
        pick[:, :upto - stored] = torch.arange(stored, upto, device="cuda")      # every new key, and repeats of any
        pick = torch.stack([p[torch.randperm(size, device="cuda", generator=g)] for p in pick])
        flags = [torch.full((size,), 7, dtype=torch.uint8, device="cuda") for _ in range(count)]
        items = [(i, keys[i][pick[i]].contiguous(), flags[i]) for i in range(count)]
        ht.ht_multi_find_or_put([t.handle for t in tabs], items)
        for i in range(count):
            new = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, pick[i], flags[i].to(torch.int64))
            at = torch.arange(n, device="cuda")
            assert torch.equal(new, ((at >= stored) & (at < upto)).to(torch.int64))
        stored = upto
        assert [t.size() for t in tabs] == [stored] * count
    assert all(t.sync() == 0 for t in tabs)
    assert all(bool(t.lookup(keys[i])[0].all()) for i, t in enumerate(tabs))
