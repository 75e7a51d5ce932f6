// Probe and claim of the GPUexplore-style bucket table (Section 4.2 of the
// paper), shared by the kernels that find-or-put or look up tiles of 32 keys:
// the single-table, multi-table, packed, fused and persistent kernels.
// The protocol and its exactly-once argument are described at the top of
// ht_bucket.cu.
#pragma once

#include "ht_multi_dev.cuh"

namespace ht {
namespace bucket {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kSec = 4;                 // slots of a 32-byte sector

// What one pass over its sector leaves of a key.
enum : uint32_t {
    kKeyDone = 0,     // found by find-or-put; not stored, for a lookup
    kKeyHit = 1,      // stored by this find-or-put; found by a lookup
    kKeyLost = 2,     // its claim lost the slot to another key: the same sector again
    kKeyFull = 3,     // its sector is full of other keys: the next one
};

// Where a key's claims start in a bucket: bits 0-7 give the sector, bits 8-15
// the slot in each sector; from there on they go around.  All kernels keep this
// order.  Any order does that is the same for all copies of a key (the argument
// in ht_bucket.cu); when every key starts at slot 0, the keys of a small
// table's batch that share a bucket all claim the same slot and all but one
// lose and try again: 16,384 new keys into 62,500 slots took 22 us, now 10.
__device__ __forceinline__ uint32_t claim_rot(uint64_t key) {
    return (uint32_t(key) ^ uint32_t(key >> 32)) * 0x9E3779B1u >> 16;
}

// The first bit set of an N-bit mask (N a power of two) from bit `from` on,
// around its end.
template <int N>
__device__ __forceinline__ uint32_t first_from(uint32_t mask, uint32_t from) {
    const uint32_t up = mask >> from;
    return up ? from + __ffs(up) - 1 : __ffs(mask) - 1;
}

// The sector (4-slot index into the table) where key's search of bucket bkt
// starts, and the one after `sec`: around the bucket's NS sectors.
template <int NS>
__device__ __forceinline__ uint64_t first_sector(uint64_t key, uint64_t bkt) {
    return bkt * NS + claim_rot(key) % NS;
}
template <int NS>
__device__ __forceinline__ uint64_t next_sector(uint64_t sec) {
    return (sec & ~uint64_t(NS - 1)) | ((sec + 1) & (NS - 1));
}

// N slot words (whole sectors), read through L2 (the table is written by
// atomics, so L1 copies would be stale) 32 bytes a load; zeros where !ok.  The
// predicate sits at each load: a branch around them makes each round of a tile
// wait for its own loads (lookups in 500 MB 665 us instead of 509).
template <int N>
__device__ __forceinline__ void load_sectors(const uint64_t* p, bool ok, uint64_t (&w)[N]) {
#pragma unroll
    for (int j = 0; j < N; j += kSec) {
        unsigned long long a = 0, b = 0, c = 0, d = 0;
        if (ok)
            asm volatile("ld.global.cg.v4.u64 {%0,%1,%2,%3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p + j));
        w[j] = a;
        w[j + 1] = b;
        w[j + 2] = c;
        w[j + 3] = d;
    }
}

// A tile of 32 keys is taken through its buckets in passes of straight-line
// code, each with one read and at most one CAS per key; keys that a pass leaves
// unsettled go to the warp's queue (Pending), which runs them 32 at a time.
// They are few, and settling them in place would stall 32 keys on the round
// trips of one or two (done so, out of line, an L2-resident replay of 10^8 keys
// took 3.7 ms; now 1.0).
//
// sector_pass: find-or-put; one lane per key reads one sector of the key's bucket with one
// 256-bit load.  A free slot in a sector ends the search: the key is in no later
// one.  At load 0.8 a stored key is found after 1.35 sectors on average, so a key
// costs a third of the words and instructions of a bucket read whole.  Bound by
// the sectors that L2 delivers (303 G/s measured; whole 128-byte buckets 92 G/s).
//
// bucket_pass: BS/8 lanes per key read its whole bucket.  For tables past L2,
// where random accesses are bound by requests that miss (40 G/s for a sector as
// for a line), and a second sector is another request that crosses to the other
// die's L2: fill of 2^27 keys 8.1 ms instead of 8.8, 20 M lookups in 500 MB 522 us
// instead of 875, BFS of 10^8 states 63 ms instead of 67.
template <int KW>
__device__ __forceinline__ uint32_t sector_pass(uint64_t* slots, uint64_t key, uint32_t val, uint64_t sec, bool ok) {
    using K = Keys<KW>;
    if (!ok) return kKeyDone;
    uint64_t* p = slots + sec * kSec;
    uint64_t w[kSec];
    load_sectors(p, true, w);
    bool hit = false;
    uint32_t e = 0;                         // free slots, slot j in bit j
#pragma unroll
    for (int j = 0; j < kSec; ++j) {
        hit |= K::keyof(w[j]) == key;
        // 64-bit keys: only EMPTY has the top bit set.
        e |= (KW == 32 ? uint32_t(K::empty(w[j])) : uint32_t(w[j] >> 63)) << j;
    }
    if (hit) return kKeyDone;
    if (!e) return kKeyFull;
    const uint64_t old =
        atomicCAS(reinterpret_cast<unsigned long long*>(p + first_from<kSec>(e, (claim_rot(key) >> 8) % kSec)), kEmpty,
                  K::word(key, val));
    return old == kEmpty ? kKeyHit : K::keyof(old) == key ? kKeyDone : kKeyLost;
}

// Bit i of x (i < 4) to bit 2i.
__device__ __forceinline__ uint32_t spread4(uint32_t x) {
    x = (x | (x << 2)) & 0x33u;
    return (x | (x << 1)) & 0x55u;
}

// Lane l holds key l (ok false without one) and a bucket's index, and gets
// back that key's status.  Group g (G lanes, 8 slots each) serves key
// q*(32/G)+g in round q.  All buckets are read up front, each round is decided
// from ballots, and the claims go out together.  ALL: lanes without a key read
// a bucket too and drop it (bkt is in range on all lanes); the compiler then
// schedules the appending kernel's loads together as well (BFS of 10^8 states
// 63 ms; 72 with predicated loads, which the others take: fill 7.83 against 7.95
// ms, lookups 509 against 575 us).
template <int KW, int BS, bool LOOKUP, bool ALL>
__device__ __forceinline__ uint32_t bucket_pass(uint64_t* slots, uint64_t mykey, uint32_t myval, uint64_t mybkt,
                                                bool myok, uint32_t* found_val = nullptr) {
    using K = Keys<KW>;
    constexpr int SPL = 8, G = BS / SPL, GPW = 32 / G, NS = BS / kSec;
    constexpr int PF = G < 2 ? G : 2;               // rounds in flight: 128 bytes of slot words per lane
    constexpr uint32_t kGMask = (1u << G) - 1u;
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
            load_sectors<SPL>(slots + at[q], ALL || ok[q], w[q]);
        }
#pragma unroll
        for (int q = 0; q < PF; ++q) {
            const int kidx = (r0 + q) * GPW + grp;
            key[q] = KW == 32 ? uint64_t(__shfl_sync(kFull, uint32_t(mykey), kidx)) : __shfl_sync(kFull, mykey, kidx);
            bool hit = false;
            uint32_t e = 0, v = 0;                  // e: free slots, slot j of the lane's share in bit j
#pragma unroll
            for (int j = SPL - 1; j >= 0; --j) {
                const bool same = K::keyof(w[q][j]) == key[q];
                hit |= same;
                if (LOOKUP && KW == 32 && same) v = K::value(w[q][j]);
                // 64-bit keys: only EMPTY has the top bit set.
                e = KW == 32 ? (e << 1) | uint32_t(K::empty(w[q][j])) : __funnelshift_l(uint32_t(w[q][j] >> 32), e, 1);
            }
            const uint32_t M = __ballot_sync(kFull, hit && ok[q]);
            const uint32_t gm = (M >> gbase) & kGMask;
            old[q] = 0;
            own[q] = false;
            if constexpr (LOOKUP) {
                const uint32_t ge = (__ballot_sync(kFull, e != 0 && ok[q]) >> gbase) & kGMask;
                full[q] = ok[q] && !gm && !ge;
                const uint32_t mm = (M >> mysh) & kGMask;
                if (myround == r0 + q) status = mm ? kKeyHit : kKeyDone;
                if (KW == 32) {
                    const uint32_t x = __shfl_sync(kFull, v, mysh + (mm ? __ffs(mm) - 1 : 0));
                    if (myround == r0 + q) *found_val = mm ? x : 0u;
                }
            } else {
                // The sectors with a free slot, and the first of them in the key's order.
                const uint32_t g0 = (__ballot_sync(kFull, (e & 15u) != 0 && ok[q]) >> gbase) & kGMask;
                const uint32_t g1 = (__ballot_sync(kFull, (e >> 4) != 0 && ok[q]) >> gbase) & kGMask;
                const uint32_t ge = spread4(g0) | (spread4(g1) << 1);
                full[q] = ok[q] && !gm && !ge;
                const uint32_t val = KW == 32 ? __shfl_sync(kFull, myval, kidx) : 0u;
                if (ok[q] && !gm && ge) {
                    const uint32_t rot = claim_rot(key[q]), sec = first_from<NS>(ge, rot % NS);
                    own[q] = uint32_t(sub) == sec / 2;
                    if (own[q]) {
                        const uint32_t j = (sec % 2) * kSec + first_from<kSec>((e >> (sec % 2 * kSec)) & 15u, (rot >> 8) % kSec);
                        old[q] = atomicCAS(reinterpret_cast<unsigned long long*>(slots + at[q] + j), kEmpty,
                                           K::word(key[q], val));
                    }
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
// first (their lines are the likeliest to be in L2 still).
constexpr int kPend = 64;
struct PendEntry {
    uint64_t key;
    uint64_t pos;      // where its answer goes
    uint64_t sec;      // the sector to try next
    uint32_t val;
    uint32_t probe;    // sectors tried: probe / NS buckets, probe % NS in the current one
};

struct Pending {
    PendEntry* q;
    uint32_t n;
    __device__ __forceinline__ explicit Pending(PendEntry* buf) : q(buf), n(0) {}
    __device__ __forceinline__ void push(bool pred, const PendEntry& d) {
        const uint32_t mask = __ballot_sync(kFull, pred);
        if (!mask) return;
        const int lane = threadIdx.x & 31;
        if (pred) q[n + __popc(mask & ((1u << lane) - 1))] = d;
        n += __popc(mask);
        __syncwarp();
    }
    // Lane l's entry of the last min(n, 32), if there is one.
    __device__ __forceinline__ bool pop(PendEntry& d) {
        const uint32_t m = n < 32u ? n : 32u;
        const uint32_t lane = threadIdx.x & 31;
        const bool have = lane < m;
        if (have) d = q[n - m + lane];
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

// Moves a key whose sector (WHOLE: bucket) was full on to the next one, of its
// next bucket after the last; false past the last bucket.
template <int NS, bool WHOLE>
__device__ __forceinline__ bool advance(const DevTable& t, PendEntry& d) {
    d.probe += WHOLE ? NS : 1;
    d.sec = next_sector<NS>(d.sec);
    if (d.probe % NS == 0) {
        const uint32_t f = d.probe / NS;
        if (f >= t.k) return false;
        d.sec = first_sector<NS>(d.key, hidx(d.key, t.seed[f], t.nbuckets));
    }
    return true;
}

// One pass of a tile (lane l holds entry d; ok false without one) against t,
// with what it leaves unsettled queued, or spilled past the last bucket.
// Returns the status of the keys that are done; `waits` on the others' lanes.
template <int KW, int BS, bool WHOLE, bool ALL>
__device__ __forceinline__ uint32_t put_pass(const DevTable& t, Pending& pend, PendEntry& d, bool ok, bool& waits) {
    constexpr int NS = BS / kSec;
    uint32_t st = WHOLE ? bucket_pass<KW, BS, false, ALL>(t.slots, d.key, d.val, d.sec / NS, ok)
                        : sector_pass<KW>(t.slots, d.key, d.val, d.sec, ok);
    waits = st >= kKeyLost;
    if (st == kKeyFull && !advance<NS, WHOLE>(t, d)) {
        st = spill_put<KW>(t, d.key, d.val);
        waits = false;
    }
    pend.push(waits, d);
    return st;
}

// The same for a lookup, a whole bucket a pass; AHEAD: a queued key's next bucket
// is touched.
template <int KW, int BS, bool AHEAD>
__device__ __forceinline__ uint32_t find_pass(const DevTable& t, Pending& pend, PendEntry& d, bool ok, bool& waits,
                                              uint32_t* val) {
    constexpr int NS = BS / kSec;
    uint32_t st = bucket_pass<KW, BS, true, false>(t.slots, d.key, 0, d.sec / NS, ok, val);
    waits = st == kKeyFull;
    if (waits && !advance<NS, true>(t, d)) {
        st = spill_find<KW>(t, d.key, val);
        waits = false;
    }
    if (AHEAD && waits) touch_l2(t.slots + d.sec / NS * BS);
    pend.push(waits, d);
    return st;
}

// Adds every lane's count to a table's size with one atomic per block: the
// last step of a kernel, reached by all its threads.
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
// are) and its new states are appended to e's states.  By sectors at every size:
// most successors are stored already and found in the first one (256 explorations of
// 440 MB together 18.8 ms; one of 49 M states, 560 MB, by sectors / whole 35.5 / 42.2
// ms at load 0.7, 41.1 / 44.6 at 0.9, 56.0 / 55.2 at 0.97).
constexpr int kMultiStage = kStageCap / 2;     // with the queues and tile map, under 48 KB a block

template <int BS>
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
    multi::StateStage<kMultiStage> stage(stage_buf);
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
    // queued at most once for each sector and slot of its k buckets.
    for (uint64_t tile = t_begin;;) {
        const bool moves = tile >= t_end || tile >= cur.b1;    // done with exploration e's tiles
        PendEntry d;
        d.key = d.pos = d.sec = 0;
        d.val = d.probe = 0;
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
            const DevTable& t = m.tables[e];
            d.sec = first_sector<BS / kSec>(d.key, hidx(d.key, t.seed[0], t.nbuckets));
        }
        bool waits;
        const uint32_t st = put_pass<64, BS, false, false>(m.tables[e], pend, d, ok, waits);
        stage.push(st == kKeyHit, d.key, m, e);
        stored += __popc(__ballot_sync(kFull, st == kKeyHit));
    }
}

}  // namespace bucket
}  // namespace ht
