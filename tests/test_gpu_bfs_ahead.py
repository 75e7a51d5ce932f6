"""Explorations whose small levels run ahead of the host: stopped at every place
relative to a group of such levels, by the level limit, a full states array and
the end, twice on one table, against the same levels made from the public
pieces (ht_successors and find-or-put, each with its own oracle tests)."""
import pytest
import torch

import paper_1712_09494_gb300 as ht
from workloads import statespace as ss

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,params", [("bucket", None), ("cuckoo", None), ("cuckoo", dict(max_batch=2048))])
@pytest.mark.parametrize("max_levels", [1, 2, 3, 4, 5, 6, 9, 4096])
def test_levels_ahead_of_the_host(scheme, params, max_levels):
    m = ss.random_model(31, C=7, L=8, R=[3, 4, 2, 5, 3, 2, 4], p_sync=0.2, P=2)
    hm = ht.make_model(m.C, m.bits, m.deg, m.tgt, m.lab, m.pairs)
    dt = torch.int32 if m.key_width == 32 else torch.int64
    t = ht.HashTable(8000, scheme, m.key_width, params)
    seen = ht.HashTable(8000, scheme, m.key_width)
    front = torch.zeros(1, dtype=dt, device="cuda")
    seen.find_or_put(front)
    want, gen = [], 0
    while len(front) and len(want) < max_levels:
        want.append(len(front))
        succ = torch.empty(100 * len(front), dtype=dt, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
        ht.ht_successors(hm, front, succ, cnt)
        gen += int(cnt)
        succ = succ[:int(cnt)]
        front = succ[seen.find_or_put(succ).bool()]
    total = sum(want) + (len(front) if len(want) == max_levels else 0)
    for _ in range(2):
        t.clear()
        states = torch.full((8000,), -1, dtype=dt, device="cuda")
        res, got = ht.ht_bfs(t.handle, hm, 0, max_levels, states)
        assert got == want and res.levels == len(want) and res.successors == gen
        assert res.states == total and res.complete == (0 if len(front) else 1)
        assert t.size() == total and len(torch.unique(states[:total])) == total
        assert bool((states[total:] == -1).all())
    # A states array that some level overflows.
    cap = max(1, total // 2)
    if cap < total:
        t.clear()
        states = torch.full((cap + 64,), -1, dtype=dt, device="cuda")
        short, got = ht.ht_bfs(t.handle, hm, 0, max_levels, states[:cap])
        assert short.complete == 0 and short.states == cap and got == want[:short.levels]
        assert bool((states[cap:] == -1).all())


@pytest.mark.parametrize("width", [32, 64])
def test_large_levels_are_reordered_by_region(width):
    """A table past L2 with levels large enough for their successors to be reordered by table region (their number
    known on the device only), every state with the most successors a state can have; against smaller tables."""
    m = ss.random_model(5, C=8, L=8, R=6, deg_lo=3, deg_hi=3)
    hm = ht.make_model(m.C, m.bits, m.deg, m.tgt, m.lab, m.pairs)
    dt = torch.int32 if width == 32 else torch.int64
    total = 6 ** 8
    runs = []
    for scheme, slots in (("bucket", 24_000_000), ("cuckoo", int(total / 0.8)), ("bucket", int(total / 0.8))):
        t = ht.HashTable(slots, scheme, width)
        states = torch.empty(total + 10, dtype=dt, device="cuda")
        res, sizes = ht.ht_bfs(t.handle, hm, 0, 4096, states)
        assert res.complete == 1 and res.states == total and t.size() == total
        at, levels = 0, []
        for n in sizes:
            levels.append(torch.sort(states[at:at + n])[0])
            at += n
        runs.append((res.successors, sizes, torch.cat(levels)))
    for r in runs[1:]:
        assert r[0] == runs[0][0] and r[1] == runs[0][1] and torch.equal(r[2], runs[0][2])
