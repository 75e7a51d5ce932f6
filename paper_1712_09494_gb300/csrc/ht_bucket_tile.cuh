// Warp-cooperative bucket probe and claim of the GPUexplore-style table
// (Section 4.2 of the paper), shared by the kernels that find-or-put or look
// up tiles of 32 keys: the single-table, multi-table, packed, fused and
// persistent kernels.
// The protocol and its exactly-once argument are described at the top of
// ht_bucket.cu.
#pragma once

#include "ht_multi_dev.cuh"

namespace ht {
namespace bucket {

constexpr unsigned kFull = 0xFFFFFFFFu;

// One lane's share of a bucket: SPL consecutive slots, read through L2
// (the table is written by atomics, so L1 copies would be stale).  Shares of
// 32 bytes or more use 256-bit loads.
template <int SPL>
__device__ __forceinline__ void load_lane(const uint64_t* p, uint64_t (&w)[SPL]) {
    if constexpr (SPL == 1) {
        w[0] = __ldcg(reinterpret_cast<const unsigned long long*>(p));
    } else if constexpr (SPL == 2) {
        const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(p));
        w[0] = v.x;
        w[1] = v.y;
    } else {
#pragma unroll
        for (int j = 0; j < SPL; j += 4) {
            unsigned long long a, b, c, d;
            asm volatile("ld.global.cg.v4.u64 {%0,%1,%2,%3}, [%4];"
                         : "=l"(a), "=l"(b), "=l"(c), "=l"(d)
                         : "l"(p + j));
            w[j] = a;
            w[j + 1] = b;
            w[j + 2] = c;
            w[j + 3] = d;
        }
    }
}

// Rounds of a tile whose buckets are read together: up to 128 bytes of slot
// words per lane in flight.
template <int G, int SPL>
struct Rounds {
    static constexpr int kCap = (16 / SPL) < 8 ? (16 / SPL) : 8;   // <= 128 B of words per lane
    static constexpr int kN = kCap < G ? kCap : G;
};

// What one pass over its bucket leaves of a key.
enum : uint32_t {
    kKeyDone = 0,     // found by find-or-put; not stored, for a lookup
    kKeyHit = 1,      // stored by this find-or-put; found by a lookup
    kKeyLost = 2,     // its claim lost the slot to another key: the same bucket again
    kKeyFull = 3,     // its bucket is full of other keys: the next hash function
};

// Where a key's claims start in a bucket's slots: claims go from there on,
// around the bucket.  Any order does that is the same for all copies of a key
// (the argument in ht_bucket.cu).  When every key starts at slot 0, the keys of
// a small table's batch that share a bucket all claim the same slot and all but
// one lose and try again: 16,384 new keys into 62,500 slots took 22 us, of which
// a batch of stored keys takes 4.
template <int BS>
__device__ __forceinline__ uint32_t claim_rot(uint64_t key) {
    return ((uint32_t(key) ^ uint32_t(key >> 32)) * 0x9E3779B1u >> 16) % uint32_t(BS);
}

// The first bit set of an N-bit mask (N a power of two) from bit `from` on,
// around its end.
template <int N>
__device__ __forceinline__ uint32_t first_from(uint32_t mask, uint32_t from) {
    const uint32_t up = mask >> from;
    return up ? from + __ffs(up) - 1 : __ffs(mask) - 1;
}

// One pass of a tile of 32 keys over one bucket each: lane l holds key l
// (ok false on lanes without one) and the index bkt of the bucket to try, and
// gets back that key's status.  Group g (G lanes) serves key q*(32/G)+g in
// round q.  The buckets of all rounds (of a chunk of rounds, for many lanes
// per key) are read up front, each round is decided from two ballots, and a
// find-or-put's claims go out together: the lane of the group that sees the
// first free slot in the key's order CASes it.  A pass is
// straight-line code, at most one bucket read and one CAS per key; keys it
// leaves unsettled go to the caller's queue (Pending below), which runs them
// 32 at a time.  They are few (a full first bucket: 1 in 25 keys over a fill
// to load 0.8, 1 in 7 at the end), so settling them inside the tile would
// stall 32 keys on the round trips of one or two; done that way, out of
// line, the calls' stack traffic alone (the table descriptor copied for each)
// was 60% of all L1 sectors, and an L2-resident replay ran at 27 G keys/s
// (now 60 and more).
template <int KW, int BS, int G, bool VALUES, bool LOOKUP>
__device__ __forceinline__ uint32_t bucket_pass(uint64_t* slots, uint64_t mykey, uint32_t myval, uint64_t mybkt,
                                                bool myok, uint32_t* found_val = nullptr) {
    using K = Keys<KW>;
    constexpr int SPL = BS / G;
    constexpr int GPW = 32 / G;
    constexpr int PF = Rounds<G, SPL>::kN;
    constexpr uint32_t kGMask = (G == 32) ? 0xFFFFFFFFu : ((1u << G) - 1u);
    static_assert(SPL >= 1 && SPL <= 8 && BS % G == 0 && G % PF == 0, "bucket/lane split");
    const int lane = threadIdx.x & 31;
    const int grp = lane / G, sub = lane % G, gbase = grp * G;
    const int mysh = (lane % GPW) * G;              // lane l's key is served by group l % GPW ...
    const int myround = lane / GPW;                 // ... in round l / GPW
    const uint32_t okmask = __ballot_sync(kFull, myok);
    const uint64_t mybase = mybkt * BS;
    uint32_t status = kKeyDone;
#pragma unroll 1
    for (int r0 = 0; r0 < G; r0 += PF) {
        uint64_t at[PF], key[PF], w[PF][SPL], old[PF];
        bool ok[PF], own[PF], full[PF];
#pragma unroll
        for (int q = 0; q < PF; ++q) {
            const int kidx = (r0 + q) * GPW + grp;
            at[q] = __shfl_sync(kFull, mybase, kidx) + uint32_t(sub * SPL);
            ok[q] = (okmask >> kidx) & 1u;
            if (ok[q]) {
                load_lane<SPL>(slots + at[q], w[q]);
            } else {
#pragma unroll
                for (int j = 0; j < SPL; ++j) w[q][j] = 0;
            }
        }
#pragma unroll
        for (int q = 0; q < PF; ++q) {
            const int kidx = (r0 + q) * GPW + grp;
            key[q] = KW == 32 ? uint64_t(__shfl_sync(kFull, uint32_t(mykey), kidx)) : __shfl_sync(kFull, mykey, kidx);
            bool hit = false;
            uint32_t e = 0, v = 0;                  // e: free slots, slot j of the lane's share in bit SPL - 1 - j
#pragma unroll
            for (int j = 0; j < SPL; ++j) {
                if constexpr (KW == 32) {
                    const bool same = uint32_t(w[q][j]) == uint32_t(key[q]);
                    hit |= same;
                    if (LOOKUP && VALUES && same) v = K::value(w[q][j]);
                    e = (e << 1) | uint32_t(uint32_t(w[q][j]) == 0xFFFFFFFFu);
                } else {
                    // Only EMPTY has the top bit set (keys reserve it).
                    hit |= w[q][j] == key[q];
                    e = __funnelshift_l(uint32_t(w[q][j] >> 32), e, 1);
                }
            }
            const uint32_t M = __ballot_sync(kFull, hit && ok[q]);
            const uint32_t E = __ballot_sync(kFull, e != 0 && ok[q]);
            const uint32_t gm = (M >> gbase) & kGMask, ge = (E >> gbase) & kGMask;
            full[q] = ok[q] && !gm && !ge;
            old[q] = 0;
            if constexpr (!LOOKUP) {
                const uint32_t rot = claim_rot<BS>(key[q]);
                own[q] = ok[q] && !gm && ge && uint32_t(sub) == first_from<G>(ge, rot / SPL);
                const uint32_t val = VALUES ? __shfl_sync(kFull, myval, kidx) : 0u;
                if (own[q]) {
                    const uint32_t j = SPL - 1 - first_from<SPL>(e, rot % SPL);
                    old[q] = atomicCAS(reinterpret_cast<unsigned long long*>(slots + at[q] + j), kEmpty,
                                       K::word(key[q], val));
                }
            } else {
                if (myround == r0 + q) status = ((M >> mysh) & kGMask) ? kKeyHit : kKeyDone;
                if (VALUES) {
                    const uint32_t mm = (M >> mysh) & kGMask;
                    const uint32_t x = __shfl_sync(kFull, v, mysh + (mm ? __ffs(mm) - 1 : 0));
                    if (myround == r0 + q) *found_val = mm ? x : 0u;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < PF; ++q) {
            const uint32_t F = __ballot_sync(kFull, full[q]);
            if constexpr (LOOKUP) {
                if (myround == r0 + q && ((F >> mysh) & 1u)) status = kKeyFull;
            } else {
                const bool stored = own[q] && old[q] == kEmpty;
                const bool lost = own[q] && !stored && K::keyof(old[q]) != key[q];
                const uint32_t S = __ballot_sync(kFull, stored);
                const uint32_t L = __ballot_sync(kFull, lost);
                if (myround == r0 + q)
                    status = ((S >> mysh) & kGMask) ? kKeyHit
                             : ((L >> mysh) & kGMask) ? kKeyLost : ((F >> mysh) & 1u) ? kKeyFull : kKeyDone;
            }
        }
    }
    return status;
}

// A warp's queue of unsettled keys in shared memory: kPend entries, of which
// at most 31 wait when a tile adds up to 32.  Taken back 32 at a time, last
// first.
constexpr int kPend = 64;
struct PendEntry {
    uint64_t key;
    uint64_t pos;      // where its answer goes
    uint32_t val;
    uint32_t f;        // the hash function to try next
};

struct Pending {
    PendEntry* q;
    uint32_t n;
    __device__ __forceinline__ explicit Pending(PendEntry* buf) : q(buf), n(0) {}
    __device__ __forceinline__ void push(bool pred, uint64_t key, uint32_t val, uint64_t pos, uint32_t f) {
        const uint32_t mask = __ballot_sync(kFull, pred);
        if (!mask) return;
        const int lane = threadIdx.x & 31;
        if (pred) {
            PendEntry& e = q[n + __popc(mask & ((1u << lane) - 1))];
            e.key = key;
            e.pos = pos;
            e.val = val;
            e.f = f;
        }
        n += __popc(mask);
        __syncwarp();
    }
    // Lane l's entry of the last min(n, 32), if there is one.
    __device__ __forceinline__ bool pop(PendEntry& e) {
        const uint32_t m = n < 32u ? n : 32u;
        const uint32_t lane = threadIdx.x & 31;
        const bool have = lane < m;
        if (have) e = q[n - m + lane];
        n -= m;
        __syncwarp();
        return have;
    }
};

// All k buckets full: the stash and the overflow set.  Out of line: rare.
template <int KW>
__device__ __noinline__ uint32_t spill_put(const DevTable& t, uint64_t key, uint32_t val) {
    return place_spill<KW>(t, key, Keys<KW>::word(key, val)) == 1 ? uint32_t(kKeyHit) : uint32_t(kKeyDone);
}

template <int KW>
__device__ __noinline__ uint32_t spill_find(const DevTable& t, uint64_t key, uint32_t* val) {
    uint64_t w = 0;
    const bool found = find_spill<KW>(t, key, __ldcg(&t.ctr->stash_used), __ldcg(&t.ctr->ovf_used), &w);
    *val = found ? Keys<KW>::value(w) : 0u;
    return found ? uint32_t(kKeyHit) : uint32_t(kKeyDone);
}

// Settles a pass's statuses: a key past its last bucket goes to the spill,
// one with a bucket left to the queue.  Returns the status of the keys that
// are done; `waits` on the lanes whose key was queued.
template <int KW>
__device__ __forceinline__ uint32_t settle_put(const DevTable& t, Pending& pend, uint32_t st, uint64_t key,
                                               uint32_t val, uint64_t pos, uint32_t f, bool& waits) {
    if (st == kKeyFull) ++f;
    if (st == kKeyFull && f >= t.k) st = spill_put<KW>(t, key, val);
    waits = st >= kKeyLost;
    pend.push(waits, key, val, pos, f);
    return st;
}

// Adds every warp's count (lane 0's) to a table's size with one atomic per
// block: the last step of a kernel, reached by all its threads.
template <int NT>
__device__ __forceinline__ void add_size(const DevTable& t, unsigned long long stored) {
    __shared__ unsigned long long s_sum[NT / 32];
    for (int o = 16; o; o >>= 1) stored += __shfl_down_sync(kFull, stored, o);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = stored;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long total = 0;
#pragma unroll
        for (int j = 0; j < NT / 32; ++j) total += s_sum[j];
        if (total) atomicAdd(&t.ctr->size, total);
    }
}

// Multi-table find-or-put of warps [gw] of [nwarps]: the step's tiles (the
// TileMap numbering of each exploration's successors) are cut into equal
// contiguous ranges, one per warp, so a warp finds its first tile's
// exploration once and then walks on in order with that exploration's
// descriptor in registers; each tile runs against exploration e's table
// (addressed as a 64-bit key table, which a 32-bit set table's words also
// are) and its new states are appended to e's states.
template <int BS, int G>
__device__ void multi_find_or_put(const MultiDev& m, const multi::TileMap& tm, uint64_t gw, uint64_t nwarps,
                                  uint64_t* stage_buf, PendEntry* pend_buf) {
    using K = Keys<64>;
    const uint64_t tiles = tm.total(m);
    const int lane = threadIdx.x & 31;
    const uint64_t per = (tiles + nwarps - 1) / nwarps;
    const uint64_t t_begin = min(tiles, gw * per), t_end = min(tiles, t_begin + per);
    if (t_begin >= t_end) return;
    // New states are staged per warp and appended, with the table's size, in
    // one atomic each when the warp moves to another exploration or the stage
    // is full: the large explorations' counters are shared by many warps.
    multi::StateStage<kStageCap> stage(stage_buf);
    Pending pend(pend_buf);
    multi::TileCursor cur;
    cur.start(m, tm, t_begin);
    uint32_t e = cur.e;
    uint64_t cnt = multi::step_count(m, e);
    unsigned long long stored = 0;
    // The next tile's keys are loaded while this one is claimed.  Lanes past
    // an exploration's count read unused words of its segment.
    uint64_t next_key = __ldcg(reinterpret_cast<const unsigned long long*>(m.succ + cur.key_index(m, t_begin, lane)));
    // Bounded: an iteration takes a tile or up to 32 queued keys, and a key is
    // queued at most once for each slot of its k buckets.
    for (uint64_t tile = t_begin;;) {
        const bool moves = tile >= t_end || tile >= cur.b1;    // done with exploration e's tiles
        PendEntry d;
        d.key = d.pos = 0;
        d.val = d.f = 0;
        bool ok;
        if (pend.n >= 32 || (moves && pend.n)) {
            ok = pend.pop(d);
        } else {
            if (moves) {
                stage.flush(m, e);
                if (lane == 0 && stored) atomicAdd(&m.tables[e].ctr->size, stored);
                stored = 0;
                if (tile >= t_end) break;
                cur.seek(m, tm, tile);
                e = cur.e;
                cnt = multi::step_count(m, e);
            }
            d.key = next_key;
            ok = 32 * (tile - cur.b0) + lane < cnt && !K::reserved(d.key);
            if (++tile < t_end) {
                multi::TileCursor nx = cur;
                nx.seek(m, tm, tile);
                next_key = __ldcg(reinterpret_cast<const unsigned long long*>(m.succ + nx.key_index(m, tile, lane)));
            }
            if (!__any_sync(kFull, ok)) continue;
        }
        const DevTable& t = m.tables[e];
        uint32_t st = bucket_pass<64, BS, G, false, false>(t.slots, d.key, 0, hidx(d.key, t.seed[d.f], t.nbuckets), ok);
        bool waits;
        st = settle_put<64>(t, pend, st, d.key, 0, 0, d.f, waits);
        stage.push(st == kKeyHit, d.key, m, e);
        stored += __popc(__ballot_sync(kFull, st == kKeyHit));
    }
}

}  // namespace bucket
}  // namespace ht
