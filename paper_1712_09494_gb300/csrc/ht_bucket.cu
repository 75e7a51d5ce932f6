// GPUexplore-style bucket table (Section 4.2 of the paper).
//
// A key hashes to a bucket of BS 8-byte slots (BS*8 = 64/128/256 bytes,
// aligned).  The bucket is read whole by BS/8 lanes, whose ballots give the
// "matches" and "free" masks (Fig. 4, steps 1-2), or a 32-byte sector at a time
// by one lane (ht_bucket_tile.cuh).  If the key is present the search stops.
// Otherwise the first free slot in the key's order of the bucket's slots is
// CASed until a CAS succeeds or returns the key itself (step 3: another key may
// take a slot between the read and the CAS).  When the bucket has no free slot
// left, the next hash function picks the next bucket; after the last one the
// key goes to the stash.
//
// Exactly-once: a slot never returns to empty and never changes its key, and
// all copies of a key claim in the same order of the slots (sector after sector
// from one that the key gives, around the bucket; in each sector from a slot
// that the key gives).  A copy that claims slot s saw every slot before it in
// that order holding another key, so a concurrent copy either meets the claimed
// word first or finds the sector (the bucket) full only after the word was
// written there; and a sector with a free slot shows the key in no sector after
// it.  A key goes
// to bucket f+1 only after bucket f was observed full without it, and
// fullness is permanent, so lookups may stop at the first non-full bucket.
#include <algorithm>

#include "ht_bucket_tile.cuh"

namespace ht {
namespace {

using namespace bucket;

// Resident blocks per SM that the kernels are compiled for: 3 for whole
// buckets (the fill of 2^27 keys takes 8.1 ms; 8.3 at 4), 5 for sectors
// (a replay of 10^8 keys 0.99 ms; 1.05 at 3 and 4, 0.98 at 6).
constexpr int kWholeBlocks = 3;
constexpr int kSectorBlocks = 5;

// find-or-put or lookup over one table.  A warp takes a fresh tile of 32 keys,
// or 32 of its queued ones when that many wait (and the rest at the end), for
// one pass; the next two tiles' keys are being loaded meanwhile.  A lookup in a
// table past L2 (AHEAD) also touches the next tile's buckets, so that its reads
// hit L2.  Past L2 bound by random 128-byte lines (40-46 G lines/s, 25 G/s where
// the line is also written): find-or-put 23 G keys/s over a fill of 2^27 keys to
// load 0.8 (19 with whole tiles settled in place), 41 on the successors of 10^8
// states (29); lookups 39 G/s (22; 31 without touching ahead, which gives
// find-or-put nothing: its claims take the time).  In L2 100 G/s (27).
template <int KW, int BS, bool VALUES, bool APPEND, bool LOOKUP, bool WHOLE, bool AHEAD>
__device__ __forceinline__ void bucket_tiles(const DevTable& t, const void* keys, const uint32_t* vals, uint64_t n,
                                             uint8_t* flags, uint32_t* out_val, typename Keys<KW>::T* new_out,
                                             unsigned long long* new_count, uint64_t new_cap) {
    using K = Keys<KW>;
    using T = typename K::T;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    unsigned long long stored = 0;
    __shared__ T s_new[APPEND ? kBlock / 32 : 1][APPEND ? kStageCap : 1];   // new keys awaiting the append
    __shared__ PendEntry s_pend[kBlock / 32][kPend];
    WarpStage<T, kStageCap> stage(s_new[APPEND ? warp : 0]);
    Pending pend(s_pend[warp]);
    uint64_t base = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) / 32 * 32;
    // This tile's key and sector, the next tile's key.
    uint64_t key0 = 0, key1 = 0;
    uint32_t val0 = 0, val1 = 0;
    auto load = [&](uint64_t i, uint64_t& key, uint32_t& val) {
        if (i >= n) return;
        key = K::load(keys, i);
        if (VALUES && !LOOKUP) val = vals[i];
    };
    load(base + lane, key0, val0);
    load(base + step + lane, key1, val1);
    auto start = [&](uint64_t key) { return first_sector<BS / kSec>(key, hidx(key, t.seed[0], t.nbuckets)); };
    uint64_t sec0 = start(key0);
    // Bounded: an iteration takes a tile or up to 32 queued keys, and a key is
    // queued at most once for each sector and slot of its k buckets.
    for (;;) {
        PendEntry d;
        bool mine, ok;
        if (pend.n >= 32 || (base >= n && pend.n)) {
            d.key = d.pos = d.sec = 0;
            d.val = d.probe = 0;
            mine = ok = pend.pop(d);
        } else if (base < n) {
            d.key = key0;
            mine = base + lane < n;
            d.pos = base + lane;
            d.sec = sec0;
            d.val = val0;
            d.probe = 0;
            ok = mine && !K::reserved(d.key);
            if (mine && !ok) set_flag(t.ctr, kFlagInvalidKey);
            key0 = key1;
            val0 = val1;
            sec0 = start(key0);
            if (AHEAD && base + step + lane < n) touch_l2(t.slots + sec0 / (BS / kSec) * BS);
            load(base + 2 * step + lane, key1, val1);
            base += step;
        } else {
            break;
        }
        uint32_t v = 0, st;
        bool waits;
        if constexpr (LOOKUP) {
            st = find_pass<KW, BS, AHEAD>(t, pend, d, ok, waits, &v);
        } else {
            st = put_pass<KW, BS, WHOLE, APPEND>(t, pend, d, ok, waits);
            stored += st == kKeyHit;
            if (APPEND) stage.push(st == kKeyHit, T(d.key), new_out, new_count, new_cap);
        }
        if (mine && !waits) {
            if (flags) flags[d.pos] = uint8_t(st);
            if (LOOKUP && VALUES) out_val[d.pos] = v;
        }
    }
    if (APPEND) stage.flush(new_out, new_count, new_cap);
    if (!LOOKUP) add_size<kBlock>(t, stored);
}

template <int KW, int BS, bool VALUES, bool APPEND, bool WHOLE>
__global__ void __launch_bounds__(kBlock, WHOLE ? kWholeBlocks : kSectorBlocks)
bucket_fop_kernel(const __grid_constant__ DevTable t, const void* __restrict__ keys, const uint32_t* __restrict__ vals,
                  uint64_t n, const unsigned long long* __restrict__ d_n, uint8_t* __restrict__ is_new,
                  typename Keys<KW>::T* __restrict__ new_out, unsigned long long* __restrict__ new_count,
                  uint64_t new_cap) {
    pdl_wait();
    if (d_n) n = min(n, uint64_t(__ldcg(d_n)));        // batch size produced on the device
    bucket_tiles<KW, BS, VALUES, APPEND, false, WHOLE, false>(t, keys, vals, n, is_new, nullptr, new_out, new_count, new_cap);
}

// Lookup: like find-or-put without claims; a bucket with a free slot ends the
// search (a key only moves on from a full bucket), all k full -> the spill.
// Buckets are read whole at every size: an absent key takes 3.1 sectors at load
// 0.8 (2^22 lookups, half absent, in L2: 78 us by sectors, 74 whole; 2^14: 17, 12).
template <int KW, int BS, bool VALUES, bool AHEAD>
__global__ void __launch_bounds__(kBlock, kWholeBlocks)
bucket_lookup_kernel(const __grid_constant__ DevTable t, const void* __restrict__ keys, uint64_t n,
                     uint32_t* __restrict__ vals, uint8_t* __restrict__ found) {
    pdl_wait();
    bucket_tiles<KW, BS, VALUES, false, true, true, AHEAD>(t, keys, nullptr, n, found, vals, nullptr, nullptr, 0);
}

// Tables past L2 have their buckets read whole (the reason and both sides' times
// are at the passes, ht_bucket_tile.cuh).
bool past_l2(const DevTable& t) { return t.nslots * 8 > l2_bytes(); }

// So have small batches in smaller tables: a warp then has one tile, and its
// unsettled keys' passes come one after another, more of them by sectors.  New
// keys to load 0.8 and stored keys, us a batch by sectors / whole: 2^14 keys
// 10.6 / 9.2 and 7.8 / 6.8, 2^18 19.9 / 17.3 and 8.8 / 10.9, 2^20 35.9 / 35.9 and
// 12.9 / 23.2, 2^22 103 / 101 and 37 / 85.
constexpr uint64_t kSectorKeys = 1ull << 19;

template <int KW, int BS, bool WHOLE>
cudaError_t launch_fop(const DevTable& t, const void* keys, const uint32_t* vals, uint64_t n,
                       const unsigned long long* d_n, uint8_t* is_new, void* new_out,
                       unsigned long long* new_count, uint64_t new_cap, cudaStream_t s, const L2Window& w) {
    using T = typename Keys<KW>::T;
    auto k = vals ? bucket_fop_kernel<KW, BS, KW == 32, false, WHOLE>
             : new_out ? bucket_fop_kernel<KW, BS, false, true, WHOLE> : bucket_fop_kernel<KW, BS, false, false, WHOLE>;
    return launch_win(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, w, t, keys, vals, n, d_n,
                      is_new, static_cast<T*>(new_out), new_count, new_cap);
}

template <int KW, int BS>
cudaError_t launch_lookup(const DevTable& t, const void* keys, uint64_t n, uint32_t* vals,
                          uint8_t* found, cudaStream_t s, const L2Window& w) {
    auto k = past_l2(t) ? (vals ? bucket_lookup_kernel<KW, BS, true, true> : bucket_lookup_kernel<KW, BS, false, true>)
                        : (vals ? bucket_lookup_kernel<KW, BS, true, false> : bucket_lookup_kernel<KW, BS, false, false>);
    return launch_win(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, w, t, keys, n, vals, found);
}

// Multi-table find-or-put of one step (the body is shared with the
// persistent kernel, bucket::multi_find_or_put).
template <int BS>
__global__ void __launch_bounds__(kBlock, 4)
multi_bucket_fop_kernel(const __grid_constant__ MultiDev m, uint64_t) {
    __shared__ uint64_t s_new[kBlock / 32][kMultiStage];
    __shared__ unsigned int s_first[multi::kExactTileExpl + 1];
    __shared__ unsigned long long s_scan[multi::kAdvShared];
    __shared__ PendEntry s_pend[kBlock / 32][kPend];
    const multi::TileMap tm = multi::tile_map<kBlock>(m, s_first, s_scan);
    const uint64_t nwarps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    const uint64_t gw = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    multi_find_or_put<BS>(m, tm, gw, nwarps, s_new[threadIdx.x >> 5], s_pend[threadIdx.x >> 5]);
}

// One warp per exploration: level 0 is the initial state.
template <int BS>
__global__ void __launch_bounds__(kBlock) multi_bucket_init_kernel(const MultiDev m) {
    const int lane = threadIdx.x & 31;
    const uint64_t nwarps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t e = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; e < m.count; e += nwarps) {
        const uint64_t key = m.s0[e];
        const bool ok = lane == 0 && !Keys<64>::reserved(key);
        const DevTable& t = m.tables[e];
        uint32_t st = kKeyDone;
        PendEntry d;
        d.key = key;
        d.val = d.probe = 0;
        d.sec = first_sector<BS / kSec>(key, hidx(key, t.seed[0], t.nbuckets));
        for (bool go = ok; go;) {               // bounded: the sectors of k buckets, each lost claim takes a slot
            st = sector_pass<64>(t.slots, key, 0, d.sec, true);
            go = st >= kKeyLost;
            if (st == kKeyFull && !advance<BS / kSec, false>(t, d)) {
                st = spill_put<64>(t, key, 0);
                go = false;
            }
        }
        __syncwarp();
        const bool my_new = st == kKeyHit;
        if (lane == 0) {
            if (ok && my_new) {
                if (m.narrow[e]) static_cast<unsigned int*>(m.states[e])[0] = static_cast<unsigned int>(key);
                else static_cast<unsigned long long*>(m.states[e])[0] = key;
                atomicAdd(&t.ctr->size, 1ull);
            }
            const unsigned long long n0 = (ok && my_new) ? 1 : 0;
            m.total[e] = n0;
            m.lo[e] = 0;
            m.hi[e] = n0;
            m.cur[e] = 0;
            m.take[e] = 0;
            m.gen[e] = 0;
            m.level[e] = 0;
            m.done[e] = n0 ? 0u : 1u;
            if (n0) m.level_sizes[e * m.max_levels] = n0;
        }
    }
}

template <int BS>
cudaError_t launch_multi(const MultiDev& m, uint64_t max_tiles, bool init, cudaStream_t s) {
    if (init) {
        auto k = multi_bucket_init_kernel<BS>;
        const int grid = int(std::min<uint64_t>(launch_blocks((const void*)k, kBlock), (m.count + 7) / 8));
        k<<<grid, kBlock, 0, s>>>(m);
    } else {
        ProfScope ps(kKBucketFop, s);
        auto k = multi_bucket_fop_kernel<BS>;
        k<<<launch_blocks((const void*)k, kBlock), kBlock, 0, s>>>(m, max_tiles);
    }
    return cudaGetLastError();
}

// Packed multi-table find-or-put (the serving loop's batches and
// ht_multi_find_or_put): the items' 32-key tiles are numbered across the
// items and each warp takes a contiguous range of them, finds its first
// tile's item once and walks the items in order, keeping the item's
// descriptor in registers and its table's size count until it moves on.
// WHOLE: buckets are read whole, for launches of few keys, by the single-table
// kernel's rule and for its reason (batches of 2^15 keys into one table of 32 MB, us
// by sectors / whole: at load 0.5 56 / 56, at 0.8 63 / 56, at 0.9 80 / 65).  In
// launches of many keys sectors are the better one to load 0.7, also past L2 (2^19
// keys into 268 MB at load 0.5 70 / 79, at 0.8 89 / 82).
template <int KW, int BS, bool WHOLE>
__global__ void __launch_bounds__(kBlock, 4)
packed_bucket_kernel(const DevTable* __restrict__ tables, const WorkDesc* __restrict__ items, uint32_t nitems,
                     uint64_t ntiles) {
    using K = Keys<KW>;
    const int lane = threadIdx.x & 31;
    const uint64_t nwarps = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    const uint64_t gw = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t per = (ntiles + nwarps - 1) / nwarps;
    const uint64_t t_begin = min(ntiles, gw * per), t_end = min(ntiles, t_begin + per);
    if (t_begin >= t_end) return;
    uint32_t r = 0, b = nitems;                        // largest r with tile_off[r] <= t_begin
    while (b - r > 1) {
        const uint32_t mid = (r + b) / 2;
        if (items[mid].tile_off <= t_begin) r = mid; else b = mid;
    }
    WorkDesc d = items[r];
    uint64_t next_off = r + 1 < nitems ? items[r + 1].tile_off : ~0ull;
    unsigned long long stored = 0;
    __shared__ PendEntry s_pend[kBlock / 32][kPend];
    Pending pend(s_pend[threadIdx.x >> 5]);
    // Bounded: an iteration takes a tile or up to 32 queued keys of the item.
    for (uint64_t tile = t_begin;;) {
        const bool moves = tile >= t_end || tile >= next_off;      // done with the item's tiles
        PendEntry p;
        p.key = p.pos = p.sec = 0;
        p.val = p.probe = 0;
        bool mine, ok;
        if (pend.n >= 32 || (moves && pend.n)) {
            mine = ok = pend.pop(p);
        } else {
            if (moves) {
                if (lane == 0 && stored) atomicAdd(&tables[d.table].ctr->size, stored);
                stored = 0;
                if (tile >= t_end) break;
                do {
                    ++r;
                    next_off = r + 1 < nitems ? items[r + 1].tile_off : ~0ull;
                } while (tile >= next_off);
                d = items[r];
            }
            p.pos = (tile - d.tile_off) * 32 + lane;
            mine = p.pos < d.n;
            p.key = mine ? K::load(d.keys, p.pos) : 0;
            ok = mine && !K::reserved(p.key);
            if (mine && !ok) set_flag(tables[d.table].ctr, kFlagInvalidKey);
            ++tile;
            const DevTable& t = tables[d.table];
            p.sec = first_sector<BS / kSec>(p.key, hidx(p.key, t.seed[0], t.nbuckets));
        }
        bool waits;
        const uint32_t st = put_pass<KW, BS, WHOLE, false>(tables[d.table], pend, p, ok, waits);
        if (mine && !waits && d.flags) d.flags[p.pos] = uint8_t(st);
        stored += __popc(__ballot_sync(kFull, st == kKeyHit));
    }
}

// One BFS level with successor generation and find-or-put fused (the
// GPUexplore way of exploring on the fly, Section 3.2): lane l of a warp
// expands frontier state l of the warp's 32; the warp lays their successors
// out in shared memory (in chunks of kFusedStage) and runs them through the
// bucket claim tile by tile; new states are appended to `out` through the
// warp's stage.  No successor buffer goes through HBM.
constexpr int kFusedBlock = 128;
constexpr int kFusedStage = 512;

template <int KW, int BS, bool WHOLE>
__global__ void __launch_bounds__(kFusedBlock, kWholeBlocks * 2)
bfs_fused_kernel(const PreparedModel* __restrict__ model, const typename Keys<KW>::T* __restrict__ frontier,
                 uint64_t n, const __grid_constant__ DevTable t, typename Keys<KW>::T* __restrict__ out,
                 unsigned long long* __restrict__ count, uint64_t cap, unsigned long long* __restrict__ gen) {
    using K = Keys<KW>;
    using T = typename K::T;
    __shared__ PreparedModel sm;
    __shared__ uint64_t s_succ[kFusedBlock / 32][kFusedStage];
    __shared__ T s_new[kFusedBlock / 32][kStageCap];
    __shared__ PendEntry s_pend[kFusedBlock / 32][kPend];
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(model);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&sm);
        for (int i = threadIdx.x; i < int(sizeof(PreparedModel) / 4); i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    uint64_t* buf = s_succ[warp];
    WarpStage<T, kStageCap> stage(s_new[warp]);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t rounds = (n + stride - 1) / stride;       // warp-uniform trip count
    unsigned long long made = 0, stored = 0;
    Pending pend(s_pend[warp]);
    // One pass over a tile of fresh successors, or over queued keys.
    auto step = [&](bool queued, uint64_t key, bool ok) {
        PendEntry d;
        d.key = key;
        d.pos = d.sec = 0;
        d.val = d.probe = 0;
        if (queued) ok = pend.pop(d);
        else d.sec = first_sector<BS / kSec>(key, hidx(key, t.seed[0], t.nbuckets));
        bool waits;
        const uint32_t res = put_pass<KW, BS, WHOLE, true>(t, pend, d, ok, waits);
        stage.push(res == kKeyHit, T(d.key), out, count, cap);
        stored += res == kKeyHit;
    };
    for (uint64_t r = 0; r < rounds; ++r) {
        const uint64_t i = r * stride + uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
        const bool act = i < n;
        const uint64_t st = act ? uint64_t(frontier[i]) : 0;
        const uint32_t cnt = act ? count_successors(sm, st) : 0;
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += v;
        }
        const uint32_t tot = __shfl_sync(kFull, incl, 31);
        const uint32_t excl = incl - cnt;
        for (uint32_t chunk = 0; chunk < tot; chunk += kFusedStage) {
            if (act && excl < chunk + kFusedStage && incl > chunk) {
                uint32_t k = excl;
                for_each_successor(sm, st, [&](uint64_t v) {
                    if (k >= chunk && k < chunk + kFusedStage) buf[k - chunk] = v;
                    ++k;
                });
            }
            __syncwarp();
            const uint32_t m = min(uint32_t(kFusedStage), tot - chunk);
            for (uint32_t j0 = 0; j0 < m || pend.n >= 32;) {
                if (pend.n >= 32) {
                    step(true, 0, false);
                } else {
                    const bool mine = j0 + lane < m;
                    const uint64_t key = mine ? buf[j0 + lane] : 0;
                    const bool ok = mine && !K::reserved(key);
                    if (mine && !ok) set_flag(t.ctr, kFlagInvalidKey);
                    step(false, key, ok);
                    j0 += 32;
                }
            }
            __syncwarp();
        }
        made += cnt;
    }
    while (pend.n) step(true, 0, false);
    stage.flush(out, count, cap);
    for (int o = 16; o; o >>= 1) made += __shfl_down_sync(kFull, made, o);
    if (lane == 0 && made) atomicAdd(gen, made);
    add_size<kFusedBlock>(t, stored);
}

// The bucket sizes that are instantiated.
#define HT_BUCKET_CONFIGS(X) X(8) X(16) X(32)

}  // namespace

cudaError_t bucket_find_or_put(const BucketCfg& c, const DevTable& t, const void* keys,
                               const uint32_t* vals, uint64_t n, const unsigned long long* d_n,
                               uint8_t* is_new, void* new_out, unsigned long long* new_count,
                               uint64_t new_cap, cudaStream_t s, const L2Window& w, bool local) {
    ProfScope ps(kKBucketFop, s);
    const bool whole = !local && (past_l2(t) || n < kSectorKeys);
#define L(KW, BS)                                                                                                    \
    return whole ? launch_fop<KW, BS, true>(t, keys, vals, n, d_n, is_new, new_out, new_count, new_cap, s, w)        \
                 : launch_fop<KW, BS, false>(t, keys, vals, n, d_n, is_new, new_out, new_count, new_cap, s, w);
#define X(BS)                                                                                                        \
    if (c.bucket_slots == BS) {                                                                                      \
        if (c.kw == 32) L(32, BS)                                                                                    \
        L(64, BS)                                                                                                    \
    }
    HT_BUCKET_CONFIGS(X)
#undef X
#undef L
    return cudaErrorInvalidValue;
}

cudaError_t multi_bucket_find_or_put(const BucketCfg& c, const MultiDev& m, uint64_t max_tiles, cudaStream_t s) {
#define X(BS)                                                                       \
    if (c.bucket_slots == BS)                                          \
        return launch_multi<BS>(m, max_tiles, false, s);
    HT_BUCKET_CONFIGS(X)
#undef X
    return cudaErrorInvalidValue;
}

cudaError_t multi_bucket_init(const BucketCfg& c, const MultiDev& m, cudaStream_t s) {
#define X(BS)                                                                       \
    if (c.bucket_slots == BS)                                          \
        return launch_multi<BS>(m, 0, true, s);
    HT_BUCKET_CONFIGS(X)
#undef X
    return cudaErrorInvalidValue;
}

cudaError_t packed_bucket_find_or_put(const BucketCfg& c, const DevTable* tables, const WorkDesc* items,
                                      uint32_t nitems, uint64_t ntiles, cudaStream_t s) {
    if (!nitems || !ntiles) return cudaSuccess;
    ProfScope ps(kKBucketFop, s);
#define L(KW, BS)                                                                                      \
    {                                                                                                     \
        auto k = ntiles * 32 < kSectorKeys ? packed_bucket_kernel<KW, BS, true>                           \
                                           : packed_bucket_kernel<KW, BS, false>;                         \
        const int grid = int(std::min<uint64_t>(launch_blocks((const void*)k, kBlock), (ntiles + 7) / 8)); \
        k<<<grid, kBlock, 0, s>>>(tables, items, nitems, ntiles);                                         \
        return cudaGetLastError();                                                                        \
    }
#define X(BS)                                                                                          \
    if (c.bucket_slots == BS) {                                                           \
        if (c.kw == 32) L(32, BS)                                                                      \
        L(64, BS)                                                                                      \
    }
    HT_BUCKET_CONFIGS(X)
#undef X
#undef L
    return cudaErrorInvalidValue;
}

cudaError_t bfs_fused_level(const BucketCfg& c, const PreparedModel* model, const void* frontier, uint64_t n,
                            const DevTable& t, void* out, unsigned long long* count, uint64_t cap,
                            unsigned long long* gen, cudaStream_t s) {
    if (!n) return cudaSuccess;
    ProfScope ps(kKBucketFop, s);
#define L(KW, BS)                                                                                     \
    {                                                                                                    \
        using T = typename Keys<KW>::T;                                                                  \
        auto k = past_l2(t) ? bfs_fused_kernel<KW, BS, true> : bfs_fused_kernel<KW, BS, false>;                                                            \
        k<<<launch_blocks((const void*)k, kFusedBlock), kFusedBlock, 0, s>>>(                            \
            model, static_cast<const T*>(frontier), n, t, static_cast<T*>(out), count, cap, gen);        \
        return cudaGetLastError();                                                                       \
    }
#define X(BS)                                                                                         \
    if (c.bucket_slots == BS) {                                                          \
        if (c.kw == 32) L(32, BS)                                                                     \
        L(64, BS)                                                                                     \
    }
    HT_BUCKET_CONFIGS(X)
#undef X
#undef L
    return cudaErrorInvalidValue;
}

cudaError_t bucket_lookup(const BucketCfg& c, const DevTable& t, const void* keys, uint64_t n,
                          uint32_t* vals, uint8_t* found, cudaStream_t s, const L2Window& w) {
    ProfScope ps(kKBucketLookup, s);
#define X(BS)                                                                  \
    if (c.bucket_slots == BS)                                                  \
        return c.kw == 32 ? launch_lookup<32, BS>(t, keys, n, vals, found, s, w) \
                          : launch_lookup<64, BS>(t, keys, n, vals, found, s, w);
    HT_BUCKET_CONFIGS(X)
#undef X
    return cudaErrorInvalidValue;
}

}  // namespace ht
