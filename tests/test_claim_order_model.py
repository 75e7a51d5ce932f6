"""Every interleaving of the bucket claims as the kernels make them, on small
models (no GPU): searches that read one sector (128-bit keys: one half) of a
bucket at a time or the whole bucket, from a place that the key gives, and the
long-key kernel's passes warp by warp.

A bucket is NS sectors of S slots.  A key's search starts in sector
order[key][0] and goes around the bucket's sectors; in a sector its claims start
at slot order[key][1] and go around.  Four searches share these rules:

    sector   one sector a pass; a free slot in it ends the search: the first
             in the key's order is claimed, and a claim lost to another key has
             the sector read again
    whole    the whole bucket a pass; the first sector in the key's order with
             a free slot is claimed in; a lost claim has the bucket read again
    half     as sector, for two-word slots that a read may show half written: a
             slot without a complete key is a candidate, which the claim's
             compare-and-swap settles, and a lost claim goes on to the next one
    wwhole   the whole bucket of two-word slots, in the same way

Each word read and each compare-and-swap is one atomic step; the checker visits
every interleaving of a few threads.  In every final state each key new to the
table was claimed by exactly one of its threads, no key is stored twice, every
sector before a key's in its order is full (what lets a later search stop at a
free slot), and a key is past a bucket only if that one is full.  Mistakes
planted in the model -- copies of a key, or searches of two kinds, that use
different orders; a lost claim taken as the end -- must be caught.
"""
import itertools

import pytest

E = "E"                                    # a word of all ones
EMPTY = (E, E)


def _around(order, n):
    return [(order + i) % n for i in range(n)]


class Buckets:
    """keys: one (low word, high word) per thread (a 64-bit key is (E, word): its slot has one word that counts); kinds:
    one search per thread; order[key]: (first sector, first slot); seq[key]: its buckets."""

    def __init__(self, keys, kinds, order, seq, NS=2, S=2, nbuckets=1, pre=None, orders=None, backward=(),
                 stop_when_lost=False):
        self.keys, self.kinds, self.seq, self.NS, self.S = list(keys), list(kinds), seq, NS, S
        self.orders = [orders[i] if orders else order[k] for i, k in enumerate(keys)]
        self.order, self.backward, self.stop_when_lost = order, backward, stop_when_lost
        slots = [EMPTY] * (NS * S * nbuckets)
        for s, k in (pre or {}).items():
            slots[s] = k
        self.pre = dict(pre or {})
        # thread state: (pc, bucket number, sector step, words read, candidates left, result)
        self.start = (tuple(slots), tuple(("read", 0, 0, (), (), None) for _ in keys))

    def _reads(self, i, f, step):
        """The words of one pass in the order that they are read: (slot, word)."""
        first, _ = self.orders[i]
        base = self.seq[self.keys[i]][f] * self.NS * self.S
        secs = range(self.NS) if self.kinds[i] in ("whole", "wwhole") else [(first + step) % self.NS]
        slots = [base + s * self.S + j for s in secs for j in range(self.S)]
        words = [(s, w) for s in slots for w in ((0, 1) if self.kinds[i] in ("half", "wwhole") else (1,))]
        return words[::-1] if i in self.backward else words

    def _candidates(self, i, f, step, seen):
        """None if the key was seen, else the slots to claim in the key's order."""
        key, kind = self.keys[i], self.kinds[i]
        first, slot0 = self.orders[i]
        base = self.seq[key][f] * self.NS * self.S
        secs = _around(first, self.NS) if kind in ("whole", "wwhole") else [(first + step) % self.NS]
        two = kind in ("half", "wwhole")
        value = {}
        for (s, w), v in zip(self._reads(i, f, step), seen):
            value.setdefault(s, [None, None])[w] = v
        free = []
        for sec in secs:
            for j in _around(slot0, self.S):
                s = base + sec * self.S + j
                lo, hi = value[s]
                complete = (lo != E and hi != E) if two else hi != E
                if complete and (not two or lo == key[0]) and hi == key[1]:
                    return None
                if not complete:
                    free.append(s)
            if free and not two:
                break
        return tuple(free)

    def step(self, state, i):
        slots, threads = state
        pc, f, step, seen, cand, res = threads[i]
        key, kind = self.keys[i], self.kinds[i]

        def put(new, slots=slots):
            t = list(threads)
            t[i] = new
            return (slots, tuple(t))

        def onward():
            if kind in ("sector", "half") and step + 1 < self.NS:
                return put(("read", f, step + 1, (), (), None))
            if f + 1 < len(self.seq[key]):
                return put(("read", f + 1, 0, (), (), None))
            return put(("done", f, 0, (), (), "full"))

        if pc == "done":
            return None
        if pc == "read":
            words = self._reads(i, f, step)
            s, w = words[len(seen)]
            seen = seen + (slots[s][w],)
            if len(seen) < len(words):
                return put(("read", f, step, seen, (), None))
            cand = self._candidates(i, f, step, seen)
            if cand is None:
                return put(("done", f, 0, (), (), "found"))
            return put(("claim", f, step, (), cand, None)) if cand else onward()
        old = slots[cand[0]]                  # claim: compare-and-swap from EMPTY
        if old == EMPTY:
            new = list(slots)
            new[cand[0]] = key
            return put(("done", f, 0, (), (), "claimed"), tuple(new))
        if old == key:
            return put(("done", f, 0, (), (), "found"))
        if self.stop_when_lost:
            return put(("done", f, 0, (), (), "found"))
        if kind in ("sector", "whole"):       # lost: the same sector or bucket again
            return put(("read", f, step, (), (), None))
        return put(("claim", f, step, (), cand[1:], None)) if len(cand) > 1 else onward()

    def finals(self, limit=3_000_000):
        seen, out, stack = {self.start}, [], [self.start]
        while stack:
            st = stack.pop()
            moved = False
            for i in range(len(self.keys)):
                nxt = self.step(st, i)
                if nxt is None:
                    continue
                moved = True
                if nxt not in seen:
                    seen.add(nxt)
                    stack.append(nxt)
                    assert len(seen) < limit, "state space too large for the test"
            if not moved:
                out.append(st)
        return out

    def violations(self, final):
        slots, threads = final
        assert all(t[0] == "done" for t in threads)
        stored = [k for k in slots if k != EMPTY]
        out = ["a key is stored twice"] if len(stored) != len(set(stored)) else []
        per = self.NS * self.S
        for k in set(self.keys):
            res = [threads[i][5] for i in range(len(self.keys)) if self.keys[i] == k]
            if k in self.pre.values():
                want = ["found"] * len(res)
            elif k in stored:
                want = ["claimed"] + ["found"] * (len(res) - 1)
            else:
                want = ["full"] * len(res)
            if sorted(res) != sorted(want):
                out.append("key %r: %r" % (k, res))
            if k not in stored or k in self.pre.values():
                continue
            b, rest = divmod(slots.index(k), per)
            for before in self.seq[k][:self.seq[k].index(b)]:
                if EMPTY in slots[before * per:(before + 1) * per]:
                    out.append("key %r is past a bucket that is not full" % (k,))
            for sec in _around(self.order[k][0], self.NS):
                if sec == rest // self.S:
                    break
                if EMPTY in slots[b * per + sec * self.S:b * per + (sec + 1) * self.S]:
                    out.append("key %r is past a sector that is not full" % (k,))
        return out

    def bad(self):
        return [v for f in self.finals() for v in [self.violations(f)] if v]


A, B, C = (E, "a"), (E, "b"), (E, "c")                     # 64-bit keys
P, Q, R = ("x", "p"), (E, "q"), ("x", "r")                 # 128-bit keys, one with a low word of all ones
ORDER = {A: (1, 1), B: (1, 1), C: (0, 1), P: (1, 1), Q: (1, 1), R: (0, 0)}
ONE = {k: [0] for k in ORDER}
TWO = {k: [0, 1] for k in ORDER}


@pytest.mark.parametrize("kinds", list(itertools.combinations_with_replacement(["sector", "whole"], 3)))
@pytest.mark.parametrize("keys", [(A, A, A), (A, B, A), (A, A, C)])
@pytest.mark.parametrize("backward", [(), (1, 2)])
def test_one_word_slots(kinds, keys, backward):
    for order in (ORDER, {A: (0, 1), B: (1, 0), C: (0, 0)}):
        assert not Buckets(keys, kinds, order, ONE, backward=backward).bad()


@pytest.mark.parametrize("kinds", [("sector", "sector", "whole"), ("whole", "sector", "whole"), ("sector",) * 3])
def test_one_word_slots_of_a_bucket_almost_full(kinds):
    """One free slot, so that losers go on to the next bucket; and none anywhere."""
    other = [(E, "o%d" % i) for i in range(8)]
    for free in range(4):
        pre = {s: other[s] for s in range(4) if s != free}
        assert not Buckets((A, B, A), kinds, ORDER, TWO, nbuckets=2, pre=pre).bad()
    pre = {s: other[s] for s in range(8) if s != 6}
    assert not Buckets((A, B, A), kinds, ORDER, TWO, nbuckets=2, pre=pre).bad()


@pytest.mark.parametrize("kinds", [("half", "half"), ("half", "wwhole"), ("wwhole", "wwhole")])
@pytest.mark.parametrize("keys", [(P, P), (Q, Q), (P, Q), (P, R)])
@pytest.mark.parametrize("backward", [(), (1,), (0, 1)])
def test_two_word_slots(kinds, keys, backward):
    """Two threads, reads of the words in either order; an empty bucket, one with one slot left, and stored keys that
    always read as candidates."""
    ones = [(E, "o%d" % i) for i in range(8)]
    pres = [{}] + [{s: ones[s] if s % 2 else ("x", "o%d" % s) for s in range(4) if s != free} for free in range(4)]
    for pre in pres:
        assert not Buckets(keys, kinds, ORDER, TWO, nbuckets=2, pre=pre, backward=backward).bad()


def test_three_copies_in_two_word_slots():
    for kinds in (("half", "half", "wwhole"), ("wwhole", "half", "wwhole")):
        assert not Buckets((P, Q, P), kinds, ORDER, ONE, S=1, backward=(2,)).bad()


@pytest.mark.parametrize("kinds,orders", [
    (("sector", "sector"), [(0, 0), (0, 1)]),              # copies of a key start at different slots
    (("sector", "sector"), [(0, 0), (1, 0)]),              # ... in different sectors
    (("sector", "whole"), [(1, 0), (0, 0)]),               # a whole-bucket search in plain slot order
    (("half", "wwhole"), [(1, 0), (0, 0)]),
])
def test_copies_in_different_orders_are_caught(kinds, orders):
    two = kinds[0] == "half"
    k = P if two else A
    assert Buckets((k, k), kinds, {k: orders[0]}, {k: [0]}, orders=orders).bad()


@pytest.mark.parametrize("kind", ["sector", "whole", "half"])
def test_a_lost_claim_taken_as_the_end_is_caught(kind):
    k = (P, R) if kind == "half" else (A, B)
    order = {x: (0, 0) for x in k}
    assert Buckets(k, (kind, kind), order, {x: [0] for x in k}, stop_when_lost=True).bad()


class LongWarps:
    """The long-key bucket kernel's pass, two or more lanes to a warp (warps: each lane's warp).  A header is EMPTY,
    ("busy", tag) or ("ready", tag); row: the slot's key.  In a pass every lane of a warp reads its bucket's
    headers; lanes without a tag match send their first claim (from a slot that the digest gives, around the
    bucket); lanes with matches compare those that are published; the lanes with no unpublished match settle their
    claims; then the others wait for theirs, compare, and claim.  The lanes of a warp go through these steps together: a
    lane may not start a step before its warp's lanes have ended the one before.  late: another order, in which
    unpublished matches are waited for before the claims that were sent are published."""

    RANK = dict({"read": 0, "sent": 1, "match": 2, "wait": 4}, **{p: 3 for p in ("claim", "lwait", "write", "publish")},
                **{p + "+": 5 for p in ("claim", "lwait", "write", "publish")})
    LATE = dict(RANK, wait=2)

    def __init__(self, keys, warps, tag, start, seq, S=2, nbuckets=1, late=False):
        self.keys, self.warps, self.tag, self.begin, self.seq, self.S = list(keys), list(warps), tag, start, seq, S
        self.rank = self.LATE if late else self.RANK
        n = S * nbuckets
        # lane state: (pc, bucket number, headers read, slots left, matches left, unpublished ones, slot, result)
        lane = ("read", 0, (), (), (), (), None, None)
        self.start = (tuple([EMPTY] * n), tuple([None] * n), tuple(lane for _ in keys))

    def _held(self, lane):
        return lane[0].rstrip("+") in ("write", "publish")

    def step(self, state, i):
        hdr, row, lanes = state
        pc, f, seen, empty, match, busy, slot, res = lanes[i]
        if pc == "done":
            return None
        at = (f, self.rank[pc])
        for j, o in enumerate(lanes):         # the warp's lanes end a step together
            if j != i and self.warps[j] == self.warps[i] and o[0] != "done" and (o[1], self.rank[o[0]]) < at:
                return None
        key = self.keys[i]
        tag = self.tag[key]
        base = self.seq[key][f] * self.S
        hdr, row = list(hdr), list(row)
        more = "+" if pc == "wait" or pc.endswith("+") else ""      # the second turn of the claims

        def put(pc, empty=(), match=(), busy=(), slot=None, res=None, f=f, seen=()):
            t = list(lanes)
            t[i] = (pc, f, seen, empty, match, busy, slot, res)
            return (tuple(hdr), tuple(row), tuple(t))

        if pc == "read":
            seen = seen + (hdr[base + len(seen)],)
            if len(seen) < self.S:
                return put("read", seen=seen)
            m = tuple(base + s for s, h in enumerate(seen) if h != EMPTY and h[1] == tag)
            e = tuple(base + s for s in _around(self.begin[tag], self.S) if seen[s] == EMPTY)
            return put("sent" if e and not m else "match", e, m)
        if pc == "match":                     # published matches are compared, the others left for later
            if not match:
                return put("wait" if busy else "claim", empty, busy=busy)
            if hdr[match[0]][0] == "busy":
                return put("match", empty, match[1:], busy + match[:1])
            if row[match[0]] == key:
                return put("done", res="found")
            return put("match", empty, match[1:], busy)
        if pc in ("wait", "lwait", "lwait+"):
            s = busy[0] if pc == "wait" else slot
            if hdr[s][0] == "busy":
                return None
            if row[s] == key:
                return put("done", res="found")
            return put("wait" if busy[1:] else "claim" + more, empty, busy=busy[1:])
        if pc.startswith("write"):
            row[slot] = key
            return put("publish" + more, slot=slot)
        if pc.startswith("publish"):
            hdr[slot] = ("ready", tag)
            return put("done", res="claimed")
        if empty:                             # sent, claim, claim+: a compare-and-swap from EMPTY
            s = empty[0]
            old = hdr[s]
            if old == EMPTY:
                hdr[s] = ("busy", tag)
                return put("write" + more, slot=s)
            return put("lwait" + more, empty[1:], slot=s) if old[1] == tag else put("claim" + more, empty[1:])
        if f + 1 < len(self.seq[key]):
            return put("read", f=f + 1)
        return put("done", res="full")

    def run(self, limit=3_000_000):
        """(wrong final or stuck states, states in which a lane with an unpublished claim is held up by a lane of its
        warp that waits for a publish)."""
        seen, stack, wrong, held_up = {self.start}, [self.start], [], []
        while stack:
            st = stack.pop()
            nexts = [self.step(st, i) for i in range(len(self.keys))]
            held_up += [st for i, n in enumerate(nexts) if n is None and self._held(st[2][i]) and
                        any(o[0] == "wait" and w == self.warps[i] for o, w in zip(st[2], self.warps))]
            for n in nexts:
                if n is not None and n not in seen:
                    seen.add(n)
                    stack.append(n)
                    assert len(seen) < limit, "state space too large for the test"
            if not any(n is not None for n in nexts):
                hdr, row, lanes = st
                stored = [row[s] for s, h in enumerate(hdr) if h != EMPTY]
                ok = all(x[0] == "done" for x in lanes) and len(stored) == len(set(stored))
                for k in set(self.keys):
                    res = sorted(x[7] or "" for j, x in enumerate(lanes) if self.keys[j] == k)
                    ok &= res == (["claimed"] + ["found"] * (len(res) - 1) if k in stored else ["full"] * len(res))
                if not ok:
                    wrong.append(st)
        return wrong, held_up


TAG = {"a": 1, "b": 1, "c": 2, "d": 3}                      # a and b share a digest
CASES = [
    (("a", "c", "c", "a"), (0, 0, 1, 1), 2, 1),            # each warp has a key that the other claims
    (("a", "b", "a", "b"), (0, 0, 1, 1), 3, 1),
    (("a", "c", "c", "d"), (0, 0, 1, 1), 2, 2),            # a full bucket among them
    (("a", "c", "d", "c", "a"), (0, 0, 1, 1, 2), 3, 1),
]


@pytest.mark.parametrize("keys,warps,S,nb", CASES)
def test_a_long_key_claim_waits_on_nothing_before_its_publish(keys, warps, S, nb):
    seq = {k: list(range(nb)) for k in TAG}
    for start in ({1: 0, 2: 0, 3: 0}, {1: 1, 2: 0, 3: 1}):
        wrong, held_up = LongWarps(keys, warps, TAG, start, seq, S, nb).run()
        assert not wrong and not held_up


def test_a_claim_held_while_its_warp_waits_is_caught():
    """The late order gives the same answers, but a header stays busy while its owner's warp waits for another's."""
    keys, warps, S, nb = CASES[0]
    wrong, held_up = LongWarps(keys, warps, TAG, {1: 0, 2: 0, 3: 0}, {k: [0] for k in TAG}, S, nb, late=True).run()
    assert not wrong and held_up
