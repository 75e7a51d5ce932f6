"""Cases to measure: what programs that use this library have it do.

Each case is one pass of such a program through the public calls -- filling a
table in batches, looking keys up, exploring a state space, advancing many
explorations or many tables together -- from the smallest calls to tables far
larger than L2, in both schemes and all key widths.

A pass starts from an empty table where it stores keys (``clear`` is part of
it), so it can be repeated.  Repeats inside a find-or-put batch may be flagged
at any one of their places, so the fills draw their repeats from earlier
batches, where every flag has one right value; repeats inside a batch are
what the replay and the explorations consist of, and those return what is
the same for every order of the keys: sizes, level sizes, and which of many
queried keys are stored.
"""
import math

import numpy as np
import torch

import paper_1712_09494_gb300 as ht

M63 = (1 << 63) - 1
M32 = (1 << 32) - 1
MAX_LEVELS = 512


def listed():
    return [
        # A model checker's small state space: a few ten thousand keys in batches of 2^14, then a membership
        # query; calls, launches and clears count, not memory.
        dict(name="fill_small", kind="fill", scheme="bucket", width=64, n=50_000, batch=1 << 14, repeats=0.3,
             load=0.8, queries=4096),
        # The headline workload: 2^27 random 64-bit keys to load 0.8, batches of 2^24, both schemes.
        dict(name="fill_bucket_64", kind="fill", scheme="bucket", width=64, n=1 << 27, batch=1 << 24, repeats=0.25,
             load=0.8, queries=0),
        dict(name="fill_cuckoo_64", kind="fill", scheme="cuckoo", width=64, n=1 << 27, batch=1 << 24, repeats=0.25,
             load=0.8, queries=0),
        # State vectors wider than 64 bits: 16-byte slots, and 256-bit vectors behind headers.
        dict(name="fill_bucket_128", kind="fill", scheme="bucket", width=128, n=1 << 26, batch=1 << 24, repeats=0.25,
             load=0.8, queries=0),
        dict(name="fill_bucket_256", kind="fill", scheme="bucket", width=256, n=1 << 25, batch=1 << 23, repeats=0.25,
             load=0.8, queries=0),
        # A map of 2^20 (key, value) pairs at load 0.5: an L2-sized table, inserted and read back.
        dict(name="map_cuckoo_32", kind="map", scheme="cuckoo", n=1 << 20, load=0.5, queries=1 << 20),
        # Membership queries against a table far larger than L2, half of them present, a ragged number of them.
        dict(name="lookup_bucket_64", kind="lookup", scheme="bucket", width=64, n=50_000_017, load=0.8,
             queries=20_000_003),
        # The paper's random sequences (its Section 5.2): 10^8 32-bit keys, each value 100 times, in one call.
        dict(name="replay_bucket_32", kind="replay", scheme="bucket", n=100_000_000, multiplicity=100,
             queries=1 << 20),
        # Exploration of 10^8 states (12 processes, 60-bit vectors), then reachability queries.
        dict(name="bfs_bucket_large", kind="bfs", scheme="bucket", width=64, local=32, windows="555555554444", pairs=4,
             sync=0.25, fused=False, queries=1 << 22),
        # Exploration of a third of a million states: short levels, where launches and waits count.
        dict(name="bfs_cuckoo_small", kind="bfs", scheme="cuckoo", width=64, local=8, windows="4444443333", pairs=4,
             sync=0.25, fused=False, queries=1 << 14),
        # 256 explorations of uneven sizes advanced together.
        dict(name="batched_bucket", kind="batched", scheme="bucket", count=256, low=10, high=20),
        # Many small tables: each round gives every table 4096 keys in one call.
        dict(name="tables_1024", kind="tables", count=1024, slots=1 << 16, keys=4096, rounds=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _any_width(rng):
    return rng.choice([32, 64, 64, 128, 192, 256, 320, 448, 512])


def draw(rng):
    kind = rng.choice(["fill", "fill", "fill", "map", "lookup", "replay", "bfs", "bfs", "batched", "tables"])
    scheme = rng.choice(["bucket", "cuckoo"])
    if kind == "fill":
        width = _any_width(rng)
        n = _log_int(rng, 5_000, (1 << 26) * 64 // max(width, 64))
        # Batches no smaller than a 24th of the keys: one flag array is returned for each.
        batch = _log_int(rng, max(256, n // 24), max(512, n // 2))
        return dict(kind=kind, scheme=scheme, width=width, n=n, batch=batch,
                    repeats=rng.choice([0.05, 0.1, 0.25, 0.5]), load=rng.choice([0.5, 0.7, 0.8, 0.85]),
                    queries=rng.choice([0, 1000, n // 3 + 1]))
    if kind == "map":
        n = _log_int(rng, 1 << 12, 1 << 25)
        return dict(kind=kind, scheme=scheme, n=n, load=rng.choice([0.5, 0.8]), queries=_log_int(rng, 1 << 10, 1 << 24))
    if kind == "lookup":
        width = _any_width(rng)
        n = _log_int(rng, 1 << 14, (1 << 27) * 64 // max(width, 64))
        return dict(kind=kind, scheme=scheme, width=width, n=n, load=rng.choice([0.5, 0.7, 0.8, 0.85]),
                    queries=_log_int(rng, 1 << 10, (1 << 25) * 64 // max(width, 64)))
    if kind == "replay":
        return dict(kind=kind, scheme=scheme, n=_log_int(rng, 1 << 16, 100_000_000),
                    multiplicity=rng.choice([1, 2, 5, 10, 50, 100, 450, 1000]), queries=1 << 18)
    if kind == "bfs":
        wide = rng.random() < 0.2
        c = 16 if wide else rng.randint(6, 12)
        local = 32 if wide else rng.choice([8, 16, 32])
        windows = [rng.randint(2, 3 if wide else 5) for _ in range(c)]
        while math.prod(windows) > 60_000_000:
            windows[windows.index(max(windows))] -= 1
        windows = "".join(str(w) for w in windows)
        bits = c * int(math.log2(local))
        width = 32 if bits <= 31 and rng.random() < 0.5 else 64 if bits <= 63 else 128
        return dict(kind=kind, scheme=scheme, width=width, local=local, windows=windows, pairs=rng.randint(0, 6),
                    sync=0.25, fused=scheme == "bucket" and width != 128 and rng.random() < 0.4,
                    queries=_log_int(rng, 1 << 10, 1 << 20))
    if kind == "batched":
        return dict(kind=kind, scheme=scheme, count=_log_int(rng, 16, 256), low=rng.choice([8, 10]),
                    high=rng.choice([14, 17, 20]))
    keys = _log_int(rng, 64, 8192)
    return dict(kind=kind, count=_log_int(rng, 32, 1024), slots=_log_int(rng, 6 * keys, 20 * keys), keys=keys,
                rounds=rng.randint(2, 4))


# ------------------------------------------------------------------ inputs
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _rng(seed, salt):
    g = torch.Generator(device=_dev())
    g.manual_seed((seed * 1000003 + salt) & M63)
    return g


def _mix63(x, seed):
    """A bijection of [0, 2^63) on an int64 tensor: odd multiplies and xor-shifts."""
    z = (x + ((seed * 0x9E3779B97F4A7C15 + 0x632BE59BD9B4E019) & M63)) & M63
    z = (z * -0x2917014799A6026D) & M63
    z = z ^ (z >> 29)
    z = (z * -0x5F89E29B87429BD1) & M63
    z = z ^ (z >> 32)
    z = (z * -0x18FC812E5F4BD725) & M63
    return z ^ (z >> 29)


def _mix32(x, seed):
    """A permutation of [0, 2^32), re-applied where it gives the reserved 2^32 - 1, so distinct indices below
    2^32 - 1 give distinct keys; as int32 with the keys' bits."""
    s = (seed * 0x9E3779B9 + 0x85EBCA6B) & M32

    def once(z):
        z = (z + s) & M32
        z = (z * 0x7FEB352D) & M32
        z = z ^ (z >> 15)
        z = (z * 0x846CA68B) & M32
        return z ^ (z >> 16)

    z = once(x)
    z = torch.where(z == M32, once(z), z)
    return (z - ((z >> 31) << 32)).to(torch.int32)


def _keys(idx, width, seed):
    """The keys of these indices: distinct indices give distinct keys, as (n,) or (n, words)."""
    if width == 32:
        return _mix32(idx, seed)
    k = _mix63(idx, seed)
    if width == 64:
        return k
    return torch.stack([k] + [_mix63(k, seed + 1 + j) for j in range(width // 64 - 1)], dim=1).contiguous()


def _stream(case, seed):
    """Index batches of a fill and, for each place, whether its key is new: fresh keys, and repeats of keys issued
    in earlier batches, shuffled."""
    g = _rng(seed, 1)
    dev = _dev()
    out, new, issued = [], [], 0
    while issued < case["n"]:
        reps = int(case["batch"] * case["repeats"]) if issued else 0
        fresh = min(case["batch"] - reps, case["n"] - issued)
        reps = min(reps, int(fresh * case["repeats"] / max(1e-9, 1 - case["repeats"])) + 1) if reps else 0
        idx = torch.cat([torch.arange(issued, issued + fresh, device=dev),
                         torch.randint(0, max(1, issued), (reps,), device=dev, generator=g)])
        order = torch.randperm(idx.numel(), device=dev, generator=g)
        out.append(idx[order])
        new.append((order < fresh).to(torch.uint8))
        issued += fresh
    return out, new


def _queries(n, q, seed):
    """Indices of queried keys, about half of them below n (stored), and which."""
    idx = torch.randint(0, 2 * n, (q,), device=_dev(), generator=_rng(seed, 2))
    return idx, (idx < n).to(torch.uint8)


def _model(rng, local, windows, pairs, sync):
    """Transition tables of processes in parallel composition.  Process c cycles through its first windows[c] local
    states and has up to two further transitions inside that window, which pair members may have to make together;
    every combination of the windows' states is reachable."""
    c = len(windows)
    bits = np.full(c, int(math.log2(local)), dtype=np.uint8)
    deg = np.zeros((16, 32), dtype=np.uint8)
    tgt = np.zeros((16, 32, 4), dtype=np.uint8)
    lab = np.zeros((16, 32, 4), dtype=np.uint8)
    members = rng.permutation(c)[:2 * min(pairs, c // 2)].reshape(-1, 2)
    for i, w in enumerate(windows):
        deg[i, :local] = rng.integers(1, 4, size=local)
        tgt[i, :local] = rng.integers(0, w, size=(local, 4))
        tgt[i, :w, 0] = (np.arange(w) + 1) % w
        mine = np.nonzero((members == i).any(axis=1))[0]
        if len(mine):
            tied = rng.random((local, 4)) < sync
            tied[:, 0] = False
            lab[i, :local][tied] = mine[0] + 1
    return ht.make_model(c, bits, deg, tgt, lab, members)


def _vectors(windows, local, width, q, seed):
    """Random state vectors: each process in its window or just past it."""
    g = _rng(seed, 3)
    bits = int(math.log2(local))
    lo = torch.zeros(q, dtype=torch.int64, device=_dev())
    hi = torch.zeros_like(lo)
    for c, w in enumerate(windows):
        top = w if c % 4 else min(local, w + 1)
        v = torch.randint(0, top, (q,), device=_dev(), generator=g)
        at = c * bits
        if at < 64:
            lo |= v << at
        if at + bits > 64:
            hi |= v << (at - 64) if at >= 64 else v >> (64 - at)
    if width == 32:
        return lo.to(torch.int32)
    return lo if width == 64 else torch.stack([lo, hi], dim=1).contiguous()


def _windows(case):
    return [int(w) for w in case["windows"]]


def _batched_shapes(case, rng):
    """Process windows of each exploration; their products are log-uniform in 2^low..2^high."""
    shapes = []
    for _ in range(case["count"]):
        c = int(rng.integers(6, 11))
        per = 2.0 ** (rng.uniform(case["low"], case["high"]) / c)
        local = int(rng.choice([8, 16, 32]))
        shapes.append((local, [int(w) for w in np.clip(np.round(per * np.exp(rng.normal(0, 0.15, size=c))), 2, local)]))
    return shapes


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind in ("fill", "lookup"):
        s["table"] = ht.HashTable(math.ceil(case["n"] / case["load"]), case["scheme"], case["width"])
        q, _ = _queries(case["n"], case["queries"], seed)
        s["queries"] = _keys(q, case["width"], seed)
    if kind == "fill":
        s["batches"] = [_keys(b, case["width"], seed) for b in _stream(case, seed)[0]]
    elif kind == "lookup":
        step = 1 << 22
        for i in range(0, case["n"], step):
            idx = torch.arange(i, min(case["n"], i + step), device=_dev())
            s["table"].insert(_keys(idx, case["width"], seed))
        s["table"].sync()
    elif kind == "map":
        s["table"] = ht.HashTable(math.ceil(case["n"] / case["load"]), case["scheme"], 32)
        idx = torch.arange(case["n"], device=_dev())
        s["keys"] = _keys(idx, 32, seed)
        s["values"] = _mix32(idx, seed + 7)
        s["queries"] = _keys(_queries(case["n"], case["queries"], seed)[0], 32, seed)
    elif kind == "replay":
        idx, q, distinct = _replay(case, seed)
        s["table"] = ht.HashTable(math.ceil(distinct * 1.25), case["scheme"], 32)
        s["keys"] = _keys(idx, 32, seed)
        s["queries"] = _keys(q, 32, seed)
    elif kind == "bfs":
        w = _windows(case)
        rng = np.random.default_rng(seed)
        s["model"] = _model(rng, case["local"], w, case["pairs"], case["sync"])
        n = math.prod(w)
        s["table"] = ht.HashTable(math.ceil(n / 0.8), case["scheme"], case["width"])
        shape = (n + 1024, 2) if case["width"] == 128 else (n + 1024,)
        s["states"] = torch.empty(shape, dtype=torch.int32 if case["width"] == 32 else torch.int64, device=_dev())
        s["fused"] = case["fused"]
        s["queries"] = _vectors(w, case["local"], case["width"], case["queries"], seed)
    elif kind == "batched":
        rng = np.random.default_rng(seed)
        shapes = _batched_shapes(case, rng)
        models = [_model(rng, local, w, int(rng.integers(1, 5)), 0.25) for local, w in shapes]
        caps = [max(256, math.ceil(math.prod(w) / 0.7)) for _, w in shapes]
        s["many"] = ht.MultiExploration(models, [0] * len(models), caps, schemes=case["scheme"], max_levels=MAX_LEVELS)
    elif kind == "tables":
        t, k, r = case["count"], case["keys"], case["rounds"]
        idx, _ = _table_rounds(case, seed)
        keys = [_keys(i.reshape(-1), 64, seed).reshape(t, k) for i in idx]
        s["tables"] = [ht.HashTable(case["slots"], "bucket", 64) for _ in range(t)]
        s["handles"] = [x.handle for x in s["tables"]]
        s["flags"] = [torch.empty(t, k, dtype=torch.uint8, device=_dev()) for _ in range(r)]
        s["items"] = [[(i, keys[j][i], s["flags"][j][i]) for i in range(t)] for j in range(r)]
    return s


def _replay(case, seed):
    """The sequence's values and the queried ones, as indices, and how many values there are to draw from."""
    rng = max(1, round(case["n"] / case["multiplicity"]))
    g = _rng(seed, 4)
    idx = torch.randint(0, rng, (case["n"],), device=_dev(), generator=g)
    q = torch.randint(0, 2 * rng, (case["queries"],), device=_dev(), generator=g)
    return idx, q, rng


def _table_rounds(case, seed):
    """Index arrays (table, key) of each round, a quarter of them repeats of the table's earlier rounds, and which
    are new."""
    t, k = case["count"], case["keys"]
    g = _rng(seed, 5)
    own = torch.arange(t, device=_dev())[:, None] << 32
    out, new = [], []
    for r in range(case["rounds"]):
        fresh = k if r == 0 else k - k // 4
        first = 0 if r == 0 else k + (r - 1) * (k - k // 4)
        i = torch.arange(first, first + fresh, device=_dev()).expand(t, fresh)
        rep = torch.randint(0, max(1, first), (t, k - fresh), device=_dev(), generator=g)
        order = torch.randperm(k, device=_dev(), generator=g)
        out.append(own + torch.cat([i, rep], dim=1)[:, order])
        new.append((order < fresh).to(torch.uint8).expand(t, k).contiguous())
    return out, new


# ------------------------------------------------------------------ one pass
def _row(sizes):
    """Level sizes, one entry for each level there could be."""
    row = np.zeros(MAX_LEVELS, dtype=np.int64)
    row[:len(sizes)] = sizes
    return row


def run(state):
    kind = state["kind"]
    if kind == "fill":
        t = state["table"]
        t.clear()
        out = [t.find_or_put(b) for b in state["batches"]]
        if len(state["queries"]):
            out.append(t.lookup(state["queries"])[0])
        return out
    if kind == "lookup":
        return [x for x in state["table"].lookup(state["queries"]) if x is not None]
    if kind == "map":
        t = state["table"]
        t.clear()
        t.insert(state["keys"], state["values"])
        return list(t.lookup(state["queries"]))
    if kind == "replay":
        t = state["table"]
        t.clear()
        t.find_or_put(state["keys"])
        found, _ = t.lookup(state["queries"])
        return dict(size=t.size(), found=found)
    if kind == "bfs":
        t = state["table"]
        t.clear()
        res, sizes = ht.ht_bfs(t.handle, state["model"], 0, MAX_LEVELS, state["states"], fused=state["fused"])
        found, _ = t.lookup(state["queries"])
        return dict(complete=res.complete, states=res.states, successors=res.successors, levels=_row(sizes),
                    found=found)
    if kind == "batched":
        m = state["many"]
        m.reset()
        m.run(mode=0)
        got = [m.result(i) for i in range(m.count)]
        return dict(states=np.array([r["states"] for r in got]), successors=np.array([r["successors"] for r in got]),
                    levels=np.stack([_row(r["level_sizes"]) for r in got]))
    for t in state["tables"]:
        t.clear()
    for items in state["items"]:
        ht.ht_multi_find_or_put(state["handles"], items)
    return state["flags"]


def work(case):
    """Bytes: every key read and every answer written once, every slot of a table that starts empty written once, every
    key that is looked up compared with one slot.  No floating-point work."""
    kind = case["kind"]
    if kind in ("fill", "lookup"):
        b = case["width"] // 8
        slot = max(8, b)
        look = case["queries"] * (b + slot + 1)
        if kind == "lookup":
            return dict(bytes=look, flops=0)
        issued = case["n"] / max(0.01, 1 - case["repeats"])
        return dict(bytes=issued * (b + 1) + case["n"] / case["load"] * slot + look, flops=0)
    if kind == "map":
        return dict(bytes=case["n"] * 8 + case["n"] / case["load"] * 8 + case["queries"] * (4 + 8 + 5), flops=0)
    if kind == "replay":
        slots = 1.25 * case["n"] / case["multiplicity"]
        return dict(bytes=case["n"] * 5 + slots * 8 + case["queries"] * (4 + 8 + 5), flops=0)
    if kind == "bfs":
        b = case["width"] // 8
        n = math.prod(_windows(case))
        # A state is written when found, read when expanded, and stored in its slot.
        return dict(bytes=n * 2 * b + n / 0.8 * max(8, b) + case["queries"] * (b + max(8, b) + 1), flops=0)
    if kind == "batched":
        # The mean of the log-uniform sizes.
        n = case["count"] * (2.0 ** case["high"] - 2.0 ** case["low"]) / ((case["high"] - case["low"]) * math.log(2))
        return dict(bytes=n * 16 + n / 0.7 * 8, flops=0)
    t, k, r = case["count"], case["keys"], case["rounds"]
    return dict(bytes=t * k * r * 9 + t * case["slots"] * 8, flops=0)


def exact(case, seed):
    """The flags that follow from how the inputs were made; none for explorations."""
    kind = case["kind"]
    if kind == "fill":
        out = _stream(case, seed)[1]
        return out + [_queries(case["n"], case["queries"], seed)[1]] if case["queries"] else out
    if kind in ("lookup", "map"):
        q, found = _queries(case["n"], case["queries"], seed)
        if kind == "lookup" and case["width"] != 32:
            return [found]
        stored = _mix32(q, seed + 7) if kind == "map" else torch.zeros(q.numel(), dtype=torch.int32, device=_dev())
        return [found, torch.where(found != 0, stored, torch.zeros_like(stored))]
    if kind == "replay":
        idx, q, distinct = _replay(case, seed)
        seen = torch.zeros(2 * distinct, dtype=torch.uint8, device=_dev())
        seen[idx] = 1
        return dict(size=int(seen.sum()), found=seen[q])
    if kind == "tables":
        return _table_rounds(case, seed)[1]
    return None
