"""Device memory that a table keeps for reordering large batches: no more than its slots take."""
import pytest
import torch

import paper_1712_09494_gb300 as ht
from workloads import device_keys as dk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,kw", [("bucket", 32), ("bucket", 64), ("bucket", 128), ("cuckoo", 64)])
def test_scratch_stays_within_the_tables_size(scheme, kw):
    slots = 17_500_000 if kw < 128 else 8_750_000       # 140 MB, a little more than L2
    n, m = int(slots * 0.8), 1 << 24                     # distinct keys, keys of the batch
    k = dk.distinct_keys_dev(n, 3, device="cuda")
    if kw == 32:
        x = dk.mix32_perm_dev(torch.arange(n, device="cuda"), 3)
        k = (x - ((x >> 31) << 32)).to(torch.int32)
    elif kw == 128:
        k = torch.stack([dk.mix63_perm_dev(k, 4), k], dim=1).contiguous()
    idx = torch.arange(m, device="cuda") % n
    batch = k[idx]
    t = ht.HashTable(slots, scheme, kw)
    flags = torch.empty(m, dtype=torch.uint8, device="cuda")
    ht.ht_find_or_put(t.handle, batch[:1000], flags[:1000])      # the kernels are loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ht.ht_find_or_put(t.handle, batch, flags)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    assert taken <= (140 + 32) * 1_000_000                       # the pool grows 32 MB at a time
    new = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, idx, flags.to(torch.int64))
    assert torch.equal(new, (torch.arange(n, device="cuda") >= 1000).to(torch.int64)) and t.size() == n
    ht.ht_find_or_put(t.handle, batch.flip(0).contiguous(), flags)
    assert not bool(flags.any()) and t.sync() == 0 and t.size() == n
