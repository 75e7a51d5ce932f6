// Tables of long keys: W = 3..8 64-bit words (192 to 512 bits).  These are
// GPUexplore's multi-word state vectors (Sections 3.2, 4.2) past what one
// 16-byte atomic covers, and the generalisation of Cuckoo hashing to keys of
// any length that Section 7 leaves as future work.
//
// No atomic covers a whole key, so a key cannot go from EMPTY to stored in
// one step; a reader could otherwise see part of a key (the long-element
// race of Section 4.2).  Both schemes therefore claim a short word
// atomically and keep the key's words apart from it.
//
// Bucket scheme: claim, then publish.  A bucket is 16 header words, one
// 128-byte line; the key of slot s is row s of the key store.  A header is
//     EMPTY (all ones) -> BUSY | tag (compare-and-swap claim) -> tag (release store)
// with tag = the key digest's low 62 bits and BUSY = bit 62.  The claimer
// writes the key's words between its two steps and waits on nothing there.
// A reader whose tag matches a header waits (bounded) until the header is
// published, reads it with acquire semantics and then compares the whole
// key.  Claims go over the slots read as EMPTY in an order that the digest
// gives, and a claim's compare-and-swap returns the header's true state, so the
// argument of the one-word kernels carries over unchanged: a key is claimed
// in at most one slot, and it sits in bucket h_f only if h_1 .. h_{f-1} were
// full.
//
// Cuckoo: indirection.  A slot is a 16-byte entry (digest, row); the key's
// words sit in row `row` of the key store, written once by the probe kernel
// that elects the key's winner.  Eviction chains move entries with 16-byte
// atomic exchanges and take the next position from the digest alone, so a
// chain reads no key words.  The insert kernel starts after the probe
// kernel has ended, so every row is complete before an entry points to it.
//
// Key-store rows hold the key's words and, for an odd word count, a zero
// word, so every row is 16-byte aligned and is read and written with 16-byte
// accesses.
#include "ht_bucket_tile.cuh"

namespace ht {
namespace {

constexpr uint64_t kBusy = 1ull << 62;
constexpr uint64_t kTagMask = kBusy - 1;
constexpr unsigned kFullMask = 0xFFFFFFFFu;
constexpr int kLBS = int(kLongBucketSlots);

struct LongWinner {
    uint64_t digest;
    uint64_t row;
    uint64_t spos;     // its entry in the claim set, cleared by the insert
    uint64_t start;    // the hash index its eviction chain starts at
};
static_assert(sizeof(LongWinner) == kWideWinnerBytes, "winner record size");

// The digest of a key: mix64 chained over its words, seeded with W.  Hash
// positions and tags are taken from the digest; equal digests of different
// keys are told apart by comparing the words.
__device__ __forceinline__ uint64_t digest_of(const uint64_t (&k)[kLongMaxWords], uint32_t W, uint64_t mask) {
    uint64_t h = mix64(0x9E3779B97F4A7C15ull * (W + 1));
#pragma unroll
    for (uint32_t j = 0; j < kLongMaxWords; ++j)
        if (j < W) h = mix64(h ^ k[j]);
    return h & mask;
}

__device__ __forceinline__ void load_key(const uint64_t* __restrict__ keys, uint64_t i, uint32_t W,
                                         uint64_t (&k)[kLongMaxWords]) {
    const uint64_t* p = keys + i * W;
#pragma unroll
    for (uint32_t j = 0; j < kLongMaxWords; ++j) k[j] = j < W ? __ldg(p + j) : 0;
}

// A key of the input batch (W words, 8-byte aligned) against k.
__device__ __forceinline__ bool input_equals(const uint64_t* row, const uint64_t (&k)[kLongMaxWords], uint32_t W) {
    bool eq = true;
#pragma unroll
    for (uint32_t j = 0; j < kLongMaxWords; ++j)
        if (j < W) eq &= __ldg(row + j) == k[j];
    return eq;
}

// A key-store row (RW words, 16-byte aligned; a padding word is 0, as in k)
// against k, with 16-byte loads.
__device__ __forceinline__ bool row_equals(const uint64_t* row, const uint64_t (&k)[kLongMaxWords], uint32_t RW) {
    bool eq = true;
#pragma unroll
    for (uint32_t j = 0; j < kLongMaxWords; j += 2)
        if (j < RW) {
            const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(row + j));
            eq &= v.x == k[j] && v.y == k[j + 1];
        }
    return eq;
}

__device__ __forceinline__ uint64_t ld_acquire(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(uint64_t* p, uint64_t v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The digest of the W words at p, without keeping them.
__device__ __forceinline__ uint64_t digest_at(const uint64_t* __restrict__ p, uint32_t W, uint64_t mask) {
    uint64_t h = mix64(0x9E3779B97F4A7C15ull * (W + 1));
#pragma unroll
    for (uint32_t j = 0; j < kLongMaxWords; ++j)
        if (j < W) h = mix64(h ^ __ldg(p + j));
    return h & mask;
}

// A key-store row against the W words of an input key, with 16-byte loads of
// the row (a padding word is not compared).
__device__ __forceinline__ bool row_is(const uint64_t* row, const uint64_t* __restrict__ key, uint32_t W) {
    bool eq = true;
#pragma unroll
    for (uint32_t j = 0; j < kLongMaxWords; j += 2)
        if (j < W) {
            const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(row + j));
            eq &= v.x == __ldg(key + j);
            if (j + 1 < W) eq &= v.y == __ldg(key + j + 1);
        }
    return eq;
}

// Bucket scheme: does slot `slot`, whose header carries the key's tag, hold
// the key?  Waits until the header is published (bounded: after
// t.spin_limit polls the timeout flag is set and the slot is taken as
// another key's).
__device__ bool slot_holds(const DevTable& t, uint64_t slot, const uint64_t* __restrict__ key, uint32_t W, uint32_t RW) {
    uint64_t h = ld_acquire(t.slots + slot);
    uint32_t spins = 0;
    while (h & kBusy) {
        if (++spins > t.spin_limit) {
            set_flag(t.ctr, kFlagTimeout);
            return false;
        }
        __nanosleep(100);
        h = ld_acquire(t.slots + slot);
    }
    return row_is(t.kstore + slot * RW, key, W);
}

__device__ __forceinline__ void store_sector(uint64_t* p, uint64_t a, uint64_t b, uint64_t c, uint64_t d) {
    asm volatile("st.global.v4.u64 [%0], {%1,%2,%3,%4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

// The words of an input key to a key-store row (a zero padding word for an
// odd W), a whole 32-byte sector a store where the row covers one: a sector
// written in two halves is missed, filled and written twice (fill of 2^25
// 256-bit keys 4.3 ms; 3.3 with whole sectors).  Rows are 4, 6 or 8 words, those
// of 6 start in the middle of a sector every second time.
__device__ __forceinline__ void copy_row(uint64_t* row, const uint64_t* __restrict__ key, uint32_t W, uint32_t RW) {
    uint64_t k[kLongMaxWords];
#pragma unroll
    for (uint32_t j = 0; j < kLongMaxWords; ++j) k[j] = j < W ? __ldg(key + j) : 0;
    if (reinterpret_cast<uintptr_t>(row) & 31) {
        *reinterpret_cast<ulonglong2*>(row) = make_ulonglong2(k[0], k[1]);
        store_sector(row + 2, k[2], k[3], k[4], k[5]);
    } else {
        store_sector(row, k[0], k[1], k[2], k[3]);
        if (RW == 6) *reinterpret_cast<ulonglong2*>(row + 4) = make_ulonglong2(k[4], k[5]);
        if (RW == 8) store_sector(row + 4, k[4], k[5], k[6], k[7]);
    }
}

// The headers of 32 buckets, one per lane (bkt; ok false without one): lane l
// gets its bucket's slots whose tag matches in bits 0-15 and its EMPTY slots
// in bits 16-31.  Two lanes read a bucket, 8 headers each with two 256-bit
// loads, 16 buckets a round; both rounds' reads go out together.
__device__ __forceinline__ uint32_t read_headers(const uint64_t* slots, uint64_t bkt, uint64_t tag, bool ok) {
    const int lane = threadIdx.x & 31, grp = lane >> 1, sub = lane & 1;
    const uint32_t okmask = __ballot_sync(kFullMask, ok);
    uint64_t w[2][8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const uint64_t b = __shfl_sync(kFullMask, bkt, q * 16 + grp);
        bucket::load_sectors<8>(slots + b * kLBS + sub * 8, (okmask >> (q * 16 + grp)) & 1u, w[q]);
    }
    uint32_t mine = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const uint64_t ot = __shfl_sync(kFullMask, tag, q * 16 + grp);
        uint32_t m = 0, e = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            m |= uint32_t((w[q][j] & ~kBusy) == ot) << j;
            e |= uint32_t(w[q][j] >> 63) << j;             // only EMPTY has the top bit set
        }
        const uint32_t x = m | (e << 16);
        const uint32_t lo = __shfl_sync(kFullMask, x, (lane & 15) * 2), hi = __shfl_sync(kFullMask, x, (lane & 15) * 2 + 1);
        if ((lane >> 4) == q) mine = lo | (hi << 8);
    }
    return ok ? mine : 0u;
}

// Bucket-scheme find-or-put (LOOKUP: lookup).  A warp takes a fresh tile of 32
// keys, one per lane, or 32 queued ones, reads one bucket of headers for each
// and settles what that bucket settles: the owner lane checks the slots whose
// tag matches, and if the key is not there and the bucket has EMPTY slots claims
// them, from one that the digest gives around the bucket, until a claim succeeds
// or another copy of the key turns up.  Keys whose bucket is full wait in the
// warp's queue for a tile of their own.  A lookup stops at the first bucket with
// an EMPTY slot, and in a table past L2 (ahead) touches the next tile's headers.
// A key's words are not kept: only a claim and a tag match read them again (from
// L1 or L2).  Bound by random lines: the headers', and the row's written or compared.
constexpr int kLongPend = 64;
struct LongEntry {
    uint64_t digest;
    uint64_t i;        // batch index
    uint32_t f;        // the hash function to try next
    uint32_t pad_;
};
// (3 blocks per SM: 3.27 ms per fill of 2^25 256-bit keys; 3.36 at 4, 4.33 with
// eight-lane reads of the buckets and the key's words held in registers.  Lookups
// in that table, half absent, run at 17.7 G/s.)
template <bool LOOKUP>
__global__ void __launch_bounds__(kBlock, 3)
long_bucket_kernel(const __grid_constant__ DevTable t, const uint64_t* __restrict__ keys, uint64_t n,
                   uint8_t* __restrict__ out, bool ahead) {
    pdl_wait();
    const uint32_t W = t.words, RW = t.row_words;
    const int lane = threadIdx.x & 31;
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    __shared__ LongEntry s_pend[kBlock / 32][kLongPend];
    LongEntry* pend = s_pend[threadIdx.x >> 5];
    uint32_t waiting = 0;
    unsigned long long added = 0;
    uint64_t base = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) / 32 * 32;
    // The next tile's digest, ready a tile ahead.
    uint64_t next_d = base + lane < n ? digest_at(keys + (base + lane) * W, W, t.digest_mask) : 0;
    // Bounded: an iteration takes a tile or up to 32 queued keys, and a key is
    // queued at most once for each of its k buckets.
    for (;;) {
        LongEntry d;
        d.digest = d.i = 0;
        d.f = d.pad_ = 0;
        bool act;
        if (waiting >= 32 || (base >= n && waiting)) {
            const uint32_t m = min(waiting, 32u);
            act = uint32_t(lane) < m;
            if (act) d = pend[waiting - m + lane];
            waiting -= m;
            __syncwarp();
        } else if (base < n) {
            d.i = base + lane;
            d.digest = next_d;
            act = d.i < n;
            base += step;
            if (base + lane < n) {
                next_d = digest_at(keys + (base + lane) * W, W, t.digest_mask);
                if (LOOKUP && ahead) touch_l2(t.slots + hidx(next_d, t.seed[0], t.nbuckets) * kLBS);
            }
        } else {
            break;
        }
        const uint64_t tag = d.digest & kTagMask;
        const uint64_t bkt = hidx(d.digest, t.seed[d.f], t.nbuckets);
        const uint32_t x = read_headers(t.slots, bkt, tag, act);
        const uint64_t slot0 = bkt * kLBS;
        const uint64_t* key = keys + d.i * W;
        uint32_t match = x & 0xFFFFu, empty = x >> 16;
        bool found = false, claimed = false;
        // The first claim of a key without a match goes out before the others'
        // matches are checked, and these rows' lines are asked for at once.
        uint64_t old = 0;
        uint32_t sl = 0;
        bool sent = !LOOKUP && !match && empty;
        if (sent) {
            sl = bucket::first_from<kLBS>(empty, uint32_t(d.digest >> 7) % kLBS);
            old = atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + slot0 + sl), kEmpty, tag | kBusy);
        }
        if (match) touch_l2(t.kstore + (slot0 + __ffs(match) - 1) * RW);
        // A match whose header is not published yet is left for later: the lanes of
        // the warp that won a claim publish theirs before any lane waits, so a wait
        // is for a lane that waits on nothing.
        uint32_t busy = 0;
        while (match && !found) {
            const uint32_t ms = __ffs(match) - 1;
            match &= match - 1;
            if (ld_acquire(t.slots + slot0 + ms) & kBusy) busy |= 1u << ms;
            else found = row_is(t.kstore + (slot0 + ms) * RW, key, W);
        }
        // Bounded: busy is empty after the first turn.
        for (;;) {
            while (!LOOKUP && empty && !busy && !found && !claimed) {
                uint64_t* hdr = t.slots + slot0 + sl;
                if (!sent) {
                    sl = bucket::first_from<kLBS>(empty, uint32_t(d.digest >> 7) % kLBS);
                    hdr = t.slots + slot0 + sl;
                    old = atomicCAS(reinterpret_cast<unsigned long long*>(hdr), kEmpty, tag | kBusy);
                }
                sent = false;
                empty &= ~(1u << sl);
                if (old == kEmpty) {
                    copy_row(t.kstore + (slot0 + sl) * RW, key, W, RW);
                    st_release(hdr, tag);
                    claimed = true;
                } else if ((old & ~kBusy) == tag) {
                    found = slot_holds(t, slot0 + sl, key, W, RW);
                }
            }
            if (!__any_sync(kFullMask, busy != 0)) break;
            while (busy && !found) {
                const uint32_t ms = __ffs(busy) - 1;
                busy &= busy - 1;
                found = slot_holds(t, slot0 + ms, key, W, RW);
            }
            busy = 0;
        }
        // A lookup's key would sit in a bucket with an EMPTY slot.
        const bool full = act && !found && !claimed && (!LOOKUP || empty == 0);
        __syncwarp();
        // Still searching: the bucket is full; the next function, if any.
        bool waits = full;
        if (full && ++d.f >= t.k) {
            waits = false;
            if (!LOOKUP) {                         // all k buckets full
                set_flag(t.ctr, kFlagDropped);
                atomicAdd(&t.ctr->dropped, 1ull);
            }
        }
        const uint32_t wm = __ballot_sync(kFullMask, waits);
        if (wm) {
            if (waits) pend[waiting + __popc(wm & ((1u << lane) - 1))] = d;
            waiting += __popc(wm);
            __syncwarp();
        }
        added += claimed;
        if (act && !waits && out) out[d.i] = uint8_t(LOOKUP ? found : claimed);
    }
    if (!LOOKUP) bucket::add_size<kBlock>(t, added);
}

// Cuckoo overflow set: linear probing over 16-byte (digest, row) entries.
__device__ int ovf_insert(const DevTable& t, uint64_t d, uint64_t row) {
    const uint32_t n = t.ovf_slots;
    uint32_t p = uint32_t(mix64(d ^ t.aux_seed) & (n - 1));
    for (uint32_t i = 0; i < n; ++i) {
        uint64_t ol, oh;
        cas128(t.ovf + 2 * uint64_t(p), d, row, ol, oh);
        if (ol == kEmpty && oh == kEmpty) return 1;
        p = (p + 1) & (n - 1);
    }
    return -1;
}

__device__ bool ovf_find(const DevTable& t, uint64_t d, const uint64_t (&k)[kLongMaxWords], uint32_t RW) {
    const uint32_t n = t.ovf_slots;
    uint32_t p = uint32_t(mix64(d ^ t.aux_seed) & (n - 1));
    for (uint32_t i = 0; i < n; ++i) {
        const ulonglong2 e = __ldcg(reinterpret_cast<const ulonglong2*>(t.ovf + 2 * uint64_t(p)));
        if (e.x == kEmpty && e.y == kEmpty) return false;
        if (e.x == d && e.y < t.kstore_rows && row_equals(t.kstore + e.y * RW, k, RW)) return true;
        p = (p + 1) & (n - 1);
    }
    return false;
}

// Cuckoo probe (LOOKUP: lookup), one thread per key.  Section 4.1: the key
// is at one of h_1 .. h_k (or in the overflow set); a chain starts at the
// first slot its probe saw EMPTY (h_1 if none), an evicted entry moves from
// h_a to h_{a+1}, and slots never return to EMPTY, so an EMPTY h_a proves
// the key absent -- and is where a new key's chain starts.  A miss claims the key's
// entry (digest, batch index) in the claim set; an entry of equal digest is
// told apart by comparing the two batch keys.  Winners wait in a per-warp
// stage in shared memory; a flush lists a stage's winners with one atomic on
// the winner count, and a winner listed at position `at` owns key-store row
// ids + at (ids: the rows handed out before this batch, advanced by the
// insert kernel), copies its words there from the batch and writes its
// record.  One atomic per flush instead of two per warp and round: those
// same-address atomics set the probe's pace when every warp issued them.
constexpr int kLongStage = 128;
struct LongStaged {
    uint64_t digest;
    uint64_t i;        // batch index
    uint64_t spos;
    uint64_t start;
};

template <bool LOOKUP>
__global__ void __launch_bounds__(kBlock)
long_cuckoo_probe_kernel(const DevTable t, const DevScratch sc, uint32_t parity, const uint64_t* __restrict__ keys,
                         uint64_t n, uint8_t* __restrict__ out) {
    pdl_wait();
    const uint32_t W = t.words, RW = t.row_words;
    const uint32_t ovf_used = __ldcg(&t.ctr->ovf_used);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t tid = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const uint64_t rounds = (n + stride - 1) / stride;      // warp-uniform trip count
    const uint64_t dseed = t.aux_seed * 3 + 1;
    const int lane = threadIdx.x & 31;
    LongWinner* win = reinterpret_cast<LongWinner*>(sc.win);
    unsigned long long probes = 0;
    constexpr int kStage = LOOKUP ? 1 : kLongStage;
    __shared__ LongStaged s_win[kBlock / 32][kStage];
    LongStaged* stage = s_win[threadIdx.x >> 5];
    uint32_t pend = 0;
    const uint64_t row_base = LOOKUP ? 0 : __ldcg(&t.ctr->ids);
    // Lists the staged winners.  A winner past the list's capacity or past
    // the key store (more keys than the table holds) gives its claim back
    // with one 16-byte atomic (other threads may be comparing against it),
    // is reported dropped and loses its flag; inside the list it leaves a
    // record with row = EMPTY that the insert kernel skips.
    auto flush = [&]() {
        __syncwarp();
        if (pend) {
            unsigned int b = 0;
            if (lane == 0) b = atomicAdd(&t.ctr->winners[parity], pend);
            b = __shfl_sync(kFullMask, b, 0);
            for (uint32_t j = lane; j < pend; j += 32) {
                const LongStaged e = stage[j];
                const uint64_t at = uint64_t(b) + j;
                const uint64_t row = row_base + at;
                const bool listed = at < sc.win_cap, stored = listed && row < t.kstore_rows;
                if (stored) copy_row(t.kstore + row * RW, keys + e.i * W, W, RW);
                if (listed) {
                    LongWinner wn;
                    wn.digest = e.digest;
                    wn.row = stored ? row : kEmpty;
                    wn.spos = e.spos;
                    wn.start = e.start;
                    win[at] = wn;
                }
                if (!stored) {
                    uint64_t ol, oh;
                    exch128(sc.set + 2 * e.spos, kEmpty, kEmpty, ol, oh);
                    set_flag(t.ctr, kFlagDropped);
                    atomicAdd(&t.ctr->dropped, 1ull);
                    if (out) out[e.i] = 0;
                }
            }
        }
        __syncwarp();
        pend = 0;
    };
    for (uint64_t r = 0; r < rounds; ++r) {
        const uint64_t i = r * stride + tid;
        const bool act = i < n;
        uint64_t k[kLongMaxWords];
        uint64_t d = 0;
        bool found = false;
        uint32_t start = 0;            // the first function whose slot was seen EMPTY (0: none)
        if (act) {
            load_key(keys, i, W, k);
            d = digest_of(k, W, t.digest_mask);
            for (uint32_t a = 0; a < t.k; ++a) {
                const ulonglong2 e =
                    __ldcg(reinterpret_cast<const ulonglong2*>(t.slots + 2 * hidx(d, t.seed[a], t.nslots)));
                ++probes;
                if (e.x == kEmpty && e.y == kEmpty) {
                    start = a;         // the key is not past it; its chain starts there
                    break;
                }
                if (e.x == d && e.y < t.kstore_rows && row_equals(t.kstore + e.y * RW, k, RW)) {
                    found = true;
                    break;
                }
            }
            if (!found && ovf_used) found = ovf_find(t, d, k, RW);
        }
        if (LOOKUP) {
            if (act && out) out[i] = uint8_t(found);
            continue;
        }
        bool winner = false;
        uint64_t spos = 0;
        if (act && !found) {
            spos = mix64(d ^ dseed) & sc.mask;
            bool settled = false;
            for (uint64_t p = 0; p <= sc.mask; ++p) {
                uint64_t ol, oh;
                cas128(sc.set + 2 * spos, d, i, ol, oh);
                if (ol == kEmpty && oh == kEmpty) {
                    winner = settled = true;
                    break;
                }
                if (ol == d && oh < n && input_equals(keys + oh * W, k, W)) {
                    settled = true;                        // another copy of the key won
                    break;
                }
                spos = (spos + 1) & sc.mask;
            }
            if (!settled) {                                // more distinct misses than the set holds
                set_flag(t.ctr, kFlagDropped);
                atomicAdd(&t.ctr->dropped, 1ull);
            }
        }
        if (act && out) out[i] = uint8_t(winner);
        const unsigned wm = __ballot_sync(kFullMask, winner);
        if (wm) {
            if (pend + __popc(wm) > uint32_t(kStage)) flush();
            if (winner) {
                LongStaged& e = stage[pend + __popc(wm & ((1u << lane) - 1))];
                e.digest = d;
                e.i = i;
                e.spos = spos;
                e.start = t.chain_h1 ? 0u : start;
            }
            pend += __popc(wm);
        }
    }
    if (!LOOKUP) {
        flush();
        for (int o = 16; o; o >>= 1) probes += __shfl_down_sync(kFullMask, probes, o);
        if (lane == 0 && probes) atomicAdd(&t.ctr->probes, probes);
    }
}

// Eviction chains of the winners' (digest, row) entries; each thread keeps
// four chains in flight and refills a chain that ends with its next winner.
__global__ void __launch_bounds__(kBlock)
long_cuckoo_insert_kernel(const DevTable t, const DevScratch sc, uint32_t parity, uint64_t max_winners) {
    constexpr int U = 4;
    pdl_wait();
    const uint64_t count = min(uint64_t(__ldcg(&t.ctr->winners[parity])), max_winners);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        t.ctr->winners[parity ^ 1u] = 0;
        // Rows ids .. ids + count - 1 went to this batch's listed winners
        // (those past the key store were dropped); no other thread of this
        // kernel reads ids, and the next probe starts after it ends.
        const unsigned long long ids = t.ctr->ids;
        t.ctr->ids = min(uint64_t(ids) + count, t.kstore_rows);
    }
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t tid = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const LongWinner* win = reinterpret_cast<const LongWinner*>(sc.win);
    unsigned long long placed = 0, exchanges = 0;
    uint64_t next = tid;
    uint64_t dg[U], row[U], pos[U];
    uint32_t evictions[U];
    bool live[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        live[u] = false;
        dg[u] = row[u] = pos[u] = 0;
        evictions[u] = 0;
    }
    // Bounded: each winner is taken once and its chain ends after at most
    // max_evictions + 1 exchanges.
    for (;;) {
        bool any = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            while (!live[u] && next < count) {
                const LongWinner wn = win[next];
                next += stride;
                if (wn.row >= t.kstore_rows) continue;     // dropped in the probe; its claim is back
                sc.set[2 * wn.spos] = kEmpty;              // leave the claim set empty for the next batch
                sc.set[2 * wn.spos + 1] = kEmpty;
                dg[u] = wn.digest;
                row[u] = wn.row;
                pos[u] = hidx(wn.digest, t.seed[wn.start < t.k ? wn.start : 0], t.nslots);
                evictions[u] = 0;
                live[u] = true;
            }
            any |= live[u];
        }
        if (!any) break;
        ulonglong2 old[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (live[u]) {
                uint64_t ol, oh;
                exch128(t.slots + 2 * pos[u], dg[u], row[u], ol, oh);
                old[u] = make_ulonglong2(ol, oh);
            }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!live[u]) continue;
            ++exchanges;
            if (old[u].x == kEmpty && old[u].y == kEmpty) {
                live[u] = false;
                ++placed;
                continue;
            }
            dg[u] = old[u].x;
            row[u] = old[u].y;
            if (++evictions[u] > t.max_evict) {
                // The chain hit the eviction bound: the held entry goes to the overflow set.
                if (ovf_insert(t, dg[u], row[u]) == 1) {
                    ++placed;
                    atomicAdd(&t.ctr->ovf_used, 1u);
                    set_flag(t.ctr, kFlagRebuild);
                } else {
                    set_flag(t.ctr, kFlagDropped);
                    atomicAdd(&t.ctr->dropped, 1ull);
                }
                live[u] = false;
                continue;
            }
            // Section 4.1: the evicted entry sat at h_a(digest) = pos, a the
            // smallest such index; it moves on to h_{a+1} (after h_k: h_1).
            uint32_t a = 0;
            for (; a + 1 < t.k; ++a)
                if (hidx(dg[u], t.seed[a], t.nslots) == pos[u]) break;
            const uint32_t nxt = (a + 1 == t.k) ? 0u : a + 1;
            pos[u] = hidx(dg[u], t.seed[nxt], t.nslots);
        }
    }
    for (int o = 16; o; o >>= 1) {
        placed += __shfl_down_sync(kFullMask, placed, o);
        exchanges += __shfl_down_sync(kFullMask, exchanges, o);
    }
    if ((threadIdx.x & 31) == 0 && placed) atomicAdd(&t.ctr->size, placed);
    if ((threadIdx.x & 31) == 0 && exchanges) atomicAdd(&t.ctr->exchanges, exchanges);
}

// Export: the rows of every published header (bucket scheme) or every
// entry of the table and the overflow set (Cuckoo), appended per warp.
__global__ void __launch_bounds__(kBlock)
long_export_kernel(const DevTable t, bool cuckoo, uint64_t* __restrict__ out, unsigned long long* __restrict__ count,
                   uint64_t cap) {
    const uint32_t W = t.words, RW = t.row_words;
    const uint64_t total = t.nslots + (cuckoo ? t.ovf_slots : 0);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t tid = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const uint64_t rounds = (total + stride - 1) / stride;
    const int lane = threadIdx.x & 31;
    for (uint64_t r = 0; r < rounds; ++r) {
        const uint64_t s = r * stride + tid;
        bool have = false;
        uint64_t src = 0;
        if (s < total) {
            if (!cuckoo) {
                const uint64_t h = __ldcg(reinterpret_cast<const unsigned long long*>(t.slots + s));
                have = (h >> 62) == 0;
                src = s;
            } else {
                const uint64_t* e = s < t.nslots ? t.slots + 2 * s : t.ovf + 2 * (s - t.nslots);
                const ulonglong2 v = __ldcg(reinterpret_cast<const ulonglong2*>(e));
                have = !(v.x == kEmpty && v.y == kEmpty);
                src = v.y;
            }
        }
        const unsigned m = __ballot_sync(kFullMask, have);
        if (!m) continue;
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(count, (unsigned long long)__popc(m));
        b = __shfl_sync(kFullMask, b, 0);
        const uint64_t at = b + __popc(m & ((1u << lane) - 1));
        if (have && at < cap && src < t.kstore_rows) {
            const uint64_t* row = t.kstore + src * RW;
            for (uint32_t j = 0; j < W; ++j) out[at * W + j] = __ldcg(reinterpret_cast<const unsigned long long*>(row + j));
        }
    }
}

}  // namespace

cudaError_t long_find_or_put(const DevTable& t, const void* keys, uint64_t n, uint8_t* is_new, cudaStream_t s) {
    if (!n) return cudaSuccess;
    ProfScope ps(kKBucketFop, s);
    auto k = long_bucket_kernel<false>;
    return launch_after(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, t, static_cast<const uint64_t*>(keys),
                        n, is_new, false);
}

cudaError_t long_lookup(const DevTable& t, const void* keys, uint64_t n, uint8_t* found, cudaStream_t s) {
    if (!n) return cudaSuccess;
    ProfScope ps(kKBucketLookup, s);
    auto k = long_bucket_kernel<true>;
    return launch_after(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, t, static_cast<const uint64_t*>(keys),
                        n, found, t.nslots * 8 > l2_bytes());
}

cudaError_t long_cuckoo_probe(const DevTable& t, const DevScratch& sc, uint32_t parity, const void* keys, uint64_t n,
                              uint8_t* is_new, cudaStream_t s) {
    ProfScope ps(kKCuckooProbe, s);
    auto k = long_cuckoo_probe_kernel<false>;
    return launch_after(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, t, sc, parity,
                        static_cast<const uint64_t*>(keys), n, is_new);
}

cudaError_t long_cuckoo_insert(const DevTable& t, const DevScratch& sc, uint32_t parity, uint64_t max_winners,
                               cudaStream_t s) {
    ProfScope ps(kKCuckooInsert, s);
    auto k = long_cuckoo_insert_kernel;
    return launch_after(k, launch_grid((const void*)k, kBlock, max_winners, kBlock), kBlock, 0, s, t, sc, parity, max_winners);
}

cudaError_t long_cuckoo_lookup(const DevTable& t, const void* keys, uint64_t n, uint8_t* found, cudaStream_t s) {
    if (!n) return cudaSuccess;
    ProfScope ps(kKCuckooLookup, s);
    DevScratch none{};
    auto k = long_cuckoo_probe_kernel<true>;
    return launch_after(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, t, none, 0u,
                        static_cast<const uint64_t*>(keys), n, found);
}

cudaError_t long_export(const DevTable& t, bool cuckoo, void* keys, unsigned long long* count, uint64_t cap,
                        cudaStream_t s) {
    ProfScope ps(kKExport, s);
    auto k = long_export_kernel;
    k<<<launch_blocks((const void*)k, kBlock), kBlock, 0, s>>>(t, cuckoo, static_cast<uint64_t*>(keys), count, cap);
    return cudaGetLastError();
}

}  // namespace ht
