// Cuckoo hashing after Alcantara et al. (Section 4.1 of the paper).
//
// Slots hold one packed 64-bit word (32-bit key | 32-bit value, or a 64-bit
// key) so a slot moves atomically.  One thread handles one key.
//
// find-or-put of a batch runs as two kernels:
//  1. probe: look each key up in its k slots h_1..h_k (and the stash).  An
//     absent key that saw an EMPTY slot stores itself at the first one with
//     a CAS from EMPTY, going on in slot order if another key took it first
//     (is_new = 1 for the copy whose CAS succeeded).  An absent key whose k
//     slots are all full claims its key in a per-batch dedup set, and the
//     single claimant per such key becomes a "winner" (is_new = 1).  Every
//     new key is appended to a compact list.
//  2. insert: each winner runs the eviction chain: exchange the word into
//     h_1; if the slot held a word k', find a with h_a(k') = slot and move
//     k' to h_{a+1}(k') (Fig. 2: key 18 evicts 26 from its h_2 slot and 26
//     moves to h_3), until an empty slot takes the word or max_evictions is
//     reached; then the stash takes it (Section 4.1: a small stash, and a
//     rebuild with new hash constants when it overflows).  Keys stored by
//     the probe are only counted here (and appended, for a frontier).
//     Section 4.1 starts every insertion at h_1 with an exchange.  Here an
//     insertion starts by default at the first of h_1..h_k that the probe
//     saw EMPTY, where it needs no eviction, and only keys with all k slots
//     full start a chain at h_1; t.chain_h1 = 1 keeps the paper's rule (a
//     CAS only at an EMPTY h_1, every other insertion a chain from h_1).
//     A Cuckoo insertion's cost is its atomics (random CASes and exchanges
//     run at the same rate whether their line is in L2 or not), so storing
//     in the probe with the one CAS that also settles duplicates takes the
//     dedup claim off most new keys.
//
// The probe stops at an empty h_1 (a key is never stored past an empty
// slot of its own).  Why that holds: slots never return to EMPTY (a CAS or
// an exchange always leaves a word), a key is stored at h_j only when
// h_1..h_(j-1) were seen occupied, and an evicted key moves from h_a to
// h_(a+1) with h_a now occupied by its evictor.
//
// Why duplicates need care: the paper's duplicate handling (Section 5.1.1:
// a thread that evicts its own key stops) does not stop a duplicate whose
// first copy was just evicted by a third key's chain, so the same key could
// be stored twice with two is_new flags.  Nothing moves a stored key during
// the probe kernel: its only table writes are CASes from EMPTY.  Copies of
// a key that store in the probe claim in slot order, so at most one CAS
// succeeds and a copy probed later finds the key; a copy that saw all k
// slots full read each after it was filled, so no copy stores the key in
// the table during the probe and the dedup set elects one winner.  Every
// winner is thus truly absent and all winners are distinct -- the
// precondition of Alcantara's insertion.
#include "ht_bucket_tile.cuh"

namespace ht {
namespace {

constexpr int kU = 4;                   // keys or eviction chains in flight per thread
constexpr int kStage = 96;              // staged winners per warp
// Resident blocks per SM that the probe with a queue is compiled for (fill of 2^27
// keys in region order 12.7 ms; 13.3 at 3, 13.5 at 5).
constexpr int kProbeBlocks = 4;

// Adds the block's per-warp sums (held by each warp's lane 0) to N table
// counters with one atomic per counter and block, not per warp: the last
// step of a kernel, reached by every thread of the block.  At one atomic per
// warp, thousands of warps ending together queued on each counter's L2
// slice, a fixed cost per launch that small launches (a BFS level's chunks)
// paid in full.
template <int N>
__device__ __forceinline__ void block_add_counters(unsigned long long* const (&dst)[N],
                                                   const unsigned long long (&v)[N]) {
    __shared__ unsigned long long s_sum[N][kBlock / 32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < N; ++c) s_sum[c][w] = v[c];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < N; ++c) {
            unsigned long long total = 0;
#pragma unroll
            for (int j = 0; j < kBlock / 32; ++j) total += s_sum[c][j];
            if (total) atomicAdd(dst[c], total);       // no return value: the adds do not wait on each other
        }
    }
}

// The start field of a winner record whose key the probe already stored.
constexpr uint32_t kStartPlaced = 0xFFFFFFFFu;

// A winner waiting in a warp's shared-memory stage: its record and its
// position in the batch (to clear its flag if the list turns out full).
struct StagedWinner {
    uint64_t word;
    uint64_t i;
    uint32_t spos;
    uint32_t start;
};

// All k slots (or one past h_1) seen without the key: the stash and overflow
// set, when in use.  Out of line: rare.
template <int KW>
__device__ __noinline__ bool spill_holds(const DevTable& t, uint64_t key, uint32_t stash_used, uint32_t ovf_used,
                                         uint64_t* w) {
    return find_spill<KW>(t, key, stash_used, ovf_used, w);
}

// A warp's stage of winners in shared memory, listed with one atomic on the
// winner count per flush, so that no pass waits on a shared counter.
template <int KW>
struct WinnerStage {
    const DevTable& t;
    const DevScratch& sc;
    uint32_t parity;
    uint8_t* out_flag;
    StagedWinner* stage;
    uint32_t pend = 0;
    __device__ WinnerStage(const DevTable& t, const DevScratch& sc, uint32_t parity, uint8_t* out_flag, StagedWinner* stage)
        : t(t), sc(sc), parity(parity), out_flag(out_flag), stage(stage) {}
    // Entries past the list's capacity (more winners than the table holds)
    // give their claim back, are reported dropped and lose their flag --
    // unless the probe stored them already.
    __device__ void flush() {
        const int lane = threadIdx.x & 31;
        __syncwarp();
        if (pend) {
            unsigned int b = 0;
            if (lane == 0) b = atomicAdd(&t.ctr->winners[parity], pend);
            b = __shfl_sync(0xFFFFFFFFu, b, 0);
            for (uint32_t j = lane; j < pend; j += 32) {
                const StagedWinner e = stage[j];
                const uint64_t at = uint64_t(b) + j;
                if (at < sc.win_cap) {
                    Winner wn;
                    wn.word = e.word;
                    wn.spos = e.spos;
                    wn.start = e.start;
                    sc.win[at] = wn;
                } else if (e.start == kStartPlaced) {
                    atomicAdd(&t.ctr->size, 1ull);     // stored already (it holds no claim)
                } else {
                    sc.set[e.spos] = kEmpty;       // no insert will clear its claim
                    set_flag(t.ctr, kFlagDropped);
                    atomicAdd(&t.ctr->dropped, 1ull);
                    if (out_flag) out_flag[e.i] = 0;
                }
            }
        }
        __syncwarp();
        pend = 0;
    }
    // Called by all lanes of the warp.
    __device__ __forceinline__ void add(bool listed, uint64_t word, uint64_t i, uint32_t spos, bool placed) {
        const unsigned wm = __ballot_sync(0xFFFFFFFFu, listed);
        if (!wm) return;
        if (pend + __popc(wm) > uint32_t(kStage)) flush();
        if (listed) {
            StagedWinner& e = stage[pend + __popc(wm & ((1u << (threadIdx.x & 31)) - 1))];
            e.word = word;
            e.i = i;
            e.spos = spos;
            e.start = placed ? kStartPlaced : 0u;
        }
        pend += __popc(wm);
    }
};

// A miss that found all k slots full goes through the claim set: the one
// claimant of each such key wins and runs an eviction chain from h_1 in the
// insert kernel.  Each CASes its key into its slot of the claim set (kept in
// L2); a slot holding another key sends it on by linear probing.
template <int KW>
__device__ __forceinline__ bool claim_key(const DevTable& t, const DevScratch& sc, uint64_t dseed, uint64_t key,
                                          uint32_t* spos) {
    const int rc = lp_insert<KW>(sc.set, uint32_t(sc.mask + 1), mix64(key ^ dseed) & sc.mask, key, key, spos);
    if (rc < 0) {                                  // more distinct misses than the table holds
        set_flag(t.ctr, kFlagDropped);
        atomicAdd(&t.ctr->dropped, 1ull);
    }
    return rc == 1;
}

// The probe's sums over the block, to the table: the last step of a kernel.
__device__ __forceinline__ void add_probe_counters(const DevTable& t, unsigned long long probes, unsigned long long misses,
                                                   unsigned long long miss_reads, unsigned long long direct,
                                                   unsigned long long stored) {
    for (int o = 16; o; o >>= 1) {
        probes += __shfl_down_sync(0xFFFFFFFFu, probes, o);
        misses += __shfl_down_sync(0xFFFFFFFFu, misses, o);
        miss_reads += __shfl_down_sync(0xFFFFFFFFu, miss_reads, o);
        direct += __shfl_down_sync(0xFFFFFFFFu, direct, o);
        stored += __shfl_down_sync(0xFFFFFFFFu, stored, o);
    }
    unsigned long long* const dst[5] = {&t.ctr->size, &t.ctr->probes, &t.ctr->probe_cas, &t.ctr->probe_misses,
                                        &t.ctr->probe_miss_reads};
    const unsigned long long sums[5] = {stored, probes, direct, misses, miss_reads};
    block_add_counters<5>(dst, sums);
}

// Probe, with the stores and the dedup.  One lane per key; a
// pass reads one slot, h_(a+1), for each key of a tile of 32 fresh keys or of 32
// that wait in the warp's queue (bucket::Pending) for their next slot: every
// lane of a pass has a slot to read, whatever the other keys' paths.  A key is
// settled by the slot that holds it or by the first EMPTY one (a key never sits
// past an empty slot of its own), 1.63 slots per key over a fill to load 0.8.
// For tables in L2 and batches in region order, where round trips are short: the
// 2^27-key fill in region order takes 7.8 instead of 10.8 ms; in L2 a replay
// of 10^8 keys of 100 occurrences takes 1.87 ms (2.16 with the kernel below).
template <int KW, bool VALUES>
__global__ void __launch_bounds__(kBlock, kProbeBlocks)
cuckoo_probe_kernel(const __grid_constant__ DevTable t, const __grid_constant__ DevScratch sc, uint32_t parity,
                    const void* __restrict__ keys, const uint32_t* __restrict__ vals, uint64_t n,
                    const unsigned long long* __restrict__ d_n, uint64_t off,
                    uint8_t* __restrict__ out_flag, bool list_stored) {
    using K = Keys<KW>;
    pdl_wait();
    if (d_n) {                                   // batch size produced on the device
        const uint64_t total = __ldcg(d_n);
        n = total > off ? min(n, total - off) : 0;
    }
    const uint32_t stash_used = __ldcg(&t.ctr->stash_used);
    const uint32_t ovf_used = __ldcg(&t.ctr->ovf_used);
    const uint64_t step = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t dseed = t.aux_seed * 3 + 1;
    const int lane = threadIdx.x & 31;
    unsigned long long probes = 0;            // slots read
    unsigned long long misses = 0, miss_reads = 0;   // keys found nowhere, and the slots they read
    unsigned long long direct = 0;            // CASes of absent keys into table slots
    unsigned long long stored = 0;            // keys stored here and not listed
    __shared__ StagedWinner s_win[kBlock / 32][kStage];
    __shared__ bucket::PendEntry s_pend[kBlock / 32][bucket::kPend];
    bucket::Pending queue(s_pend[threadIdx.x >> 5]);
    WinnerStage<KW> winners(t, sc, parity, out_flag, s_win[threadIdx.x >> 5]);
    uint64_t base = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) / 32 * 32;
    // This tile's key and slot, the next tile's key.
    uint64_t key0 = 0, key1 = 0;
    if (base + lane < n) key0 = K::load(keys, base + lane);
    if (base + step + lane < n) key1 = K::load(keys, base + step + lane);
    uint64_t slot0 = hidx(key0, t.seed[0], t.nslots);
    // Bounded: an iteration takes a tile or up to 32 queued keys, and a key is
    // queued at most k - 1 times.
    for (;;) {
        bucket::PendEntry d;
        d.val = 0;
        uint64_t at;
        bool mine, ok;
        if (queue.n >= 32 || (base >= n && queue.n)) {
            d.key = d.pos = 0;
            d.probe = 0;
            mine = ok = queue.pop(d);
            at = hidx(d.key, t.seed[d.probe], t.nslots);
        } else if (base < n) {
            d.key = key0;
            d.pos = base + lane;
            mine = d.pos < n;
            d.probe = 0;
            at = slot0;
            ok = mine && !K::reserved(d.key);
            if (mine && !ok) set_flag(t.ctr, kFlagInvalidKey);
            key0 = key1;
            slot0 = hidx(key0, t.seed[0], t.nslots);
            if (base + 2 * step + lane < n) key1 = K::load(keys, base + 2 * step + lane);
            base += step;
        } else {
            break;
        }
        uint64_t w = kEmpty;
        if (ok) w = __ldcg(reinterpret_cast<const unsigned long long*>(t.slots + at));
        probes += ok;
        bool found = ok && K::keyof(w) == d.key;
        bool miss = ok && !found && (K::empty(w) || d.probe + 1 >= t.k);
        const bool waits = ok && !found && !miss;
        if (miss && (stash_used | ovf_used) && spill_holds<KW>(t, d.key, stash_used, ovf_used, &w)) {
            found = true;
            miss = false;
        }
        if (waits) ++d.probe;
        queue.push(waits, d);
        if (miss) {
            ++misses;
            miss_reads += d.probe + 1;
        }
        // A miss that saw an EMPTY slot stores itself there with a CAS
        // from EMPTY, trying its slots in order from that one: a CAS that
        // returns the key means another copy stored it first (not new);
        // one that returns another key moves on to the next slot, which
        // the CAS reads as well.  This is the bucket scheme's claim in
        // a fixed order (Section 4.2), over h_a..h_k.  Nothing leaves a slot
        // during the probe kernel, so a key is stored in at most one slot
        // and every copy probed later finds it; a copy that saw all k
        // slots full read each after it was full, so no copy stores
        // it in the table here.  With t.chain_h1 only an EMPTY h_1 is
        // tried (Section 4.1 starts every insertion at h_1).
        bool placed = false;
        bool cas = miss && K::empty(w) && (!t.chain_h1 || d.probe == 0);
        bool claim = miss && !cas;
        while (cas) {                          // bounded: on to the next of k slots
            const uint64_t cw = atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + at), kEmpty,
                                          K::word(d.key, VALUES ? vals[d.pos] : 0u));
            ++direct;
            cas = false;
            if (cw == kEmpty) {
                placed = true;
            } else if (K::keyof(cw) == d.key) {
                // another copy stored it
            } else if (t.chain_h1 || d.probe + 1 >= t.k) {
                claim = true;                  // every slot is full now
            } else {
                ++d.probe;
                at = hidx(d.key, t.seed[d.probe], t.nslots);
                cas = true;
            }
        }
        __syncwarp();
        bool winner = placed;
        uint32_t spos = 0;
        if (claim) winner = claim_key<KW>(t, sc, dseed, d.key, &spos);
        if (mine && !waits && out_flag) out_flag[d.pos] = uint8_t(winner);
        // Keys this kernel stored are listed only for a caller that appends
        // the new keys (list_stored); otherwise they are just counted.
        stored += placed && !list_stored;
        const bool listed = winner && (list_stored || !placed);
        winners.add(listed, listed ? K::word(d.key, VALUES ? vals[d.pos] : 0u) : 0, d.pos, spos, placed);
    }
    winners.flush();
    add_probe_counters(t, probes, misses, miss_reads, direct, stored);
}

// The same with four keys per thread in lock step, one slot of each at a time
// until all are settled, then their CASes.  For tables past L2 whose batch is not
// in region order: bound by random lines, read and then claimed, of which it keeps
// 64 or 96 warps' worth in flight per SM (the queue 32).  Fills to load 0.5: 2^26
// keys in batches of 2^22 4.96 ms (5.12 with the queue), 2^27 in 2^24 10.53 (10.83).
// BLOCKS per SM: 3 while a part of the lines is found in L2, 2 past four times L2
// (cuckoo_probe), where more in flight only queue.
template <int KW, bool VALUES, int BLOCKS>
__global__ void __launch_bounds__(kBlock, BLOCKS)
cuckoo_probe_far_kernel(const __grid_constant__ DevTable t, const __grid_constant__ DevScratch sc, uint32_t parity,
                        const void* __restrict__ keys, const uint32_t* __restrict__ vals, uint64_t n,
                        const unsigned long long* __restrict__ d_n, uint64_t off, uint8_t* __restrict__ out_flag,
                        bool list_stored) {
    using K = Keys<KW>;
    pdl_wait();
    if (d_n) {                                   // batch size produced on the device
        const uint64_t total = __ldcg(d_n);
        n = total > off ? min(n, total - off) : 0;
    }
    const uint32_t stash_used = __ldcg(&t.ctr->stash_used);
    const uint32_t ovf_used = __ldcg(&t.ctr->ovf_used);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t tid = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const uint64_t rounds = (n + stride * kU - 1) / (stride * kU);     // warp-uniform trip count
    const uint64_t dseed = t.aux_seed * 3 + 1;
    unsigned long long probes = 0, misses = 0, miss_reads = 0, direct = 0, stored = 0;
    __shared__ StagedWinner s_win[kBlock / 32][kStage];
    WinnerStage<KW> winners(t, sc, parity, out_flag, s_win[threadIdx.x >> 5]);
    // The next round's keys are loaded while this round waits on the table.
    uint64_t next_key[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        const uint64_t i = uint64_t(u) * stride + tid;
        next_key[u] = i < n ? K::load(keys, i) : 0;
    }
    for (uint64_t r = 0; r < rounds; ++r) {
        uint64_t key[kU], w[kU];
        uint32_t at[kU];                         // the function whose slot was read last
        bool act[kU], found[kU], more[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            act[u] = (r * kU + u) * stride + tid < n;
            key[u] = next_key[u];
            const uint64_t j = ((r + 1) * kU + u) * stride + tid;
            if (j < n) next_key[u] = K::load(keys, j);
            if (act[u] && K::reserved(key[u])) {
                set_flag(t.ctr, kFlagInvalidKey);
                act[u] = false;
            }
            more[u] = act[u];
            found[u] = false;
            w[u] = kEmpty;
            at[u] = 0;
        }
        for (uint32_t a = 0; a < t.k; ++a) {
            bool any = false;
#pragma unroll
            for (int u = 0; u < kU; ++u) any |= more[u];
            if (!__any_sync(0xFFFFFFFFu, any)) break;
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (more[u])
                    w[u] = __ldcg(reinterpret_cast<const unsigned long long*>(t.slots + hidx(key[u], t.seed[a], t.nslots)));
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (!more[u]) continue;
                ++probes;
                at[u] = a;
                found[u] = K::keyof(w[u]) == key[u];
                more[u] = !found[u] && !K::empty(w[u]);
            }
        }
        // The CASes of the misses that saw an EMPTY slot, in slot order from it,
        // by the rules of the kernel above.
        bool placed[kU], claim[kU], cas[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const bool empty = K::empty(w[u]);
            uint64_t kept;
            if (act[u] && !found[u] && (stash_used | ovf_used))
                found[u] = spill_holds<KW>(t, key[u], stash_used, ovf_used, &kept);
            const bool miss = act[u] && !found[u];
            misses += miss;
            miss_reads += miss ? at[u] + 1 : 0;
            cas[u] = miss && empty && (!t.chain_h1 || at[u] == 0);
            claim[u] = miss && !cas[u];
            placed[u] = false;
        }
        for (uint32_t pass = 0; pass < t.k; ++pass) {
            bool any = false;
#pragma unroll
            for (int u = 0; u < kU; ++u) any |= cas[u];
            if (!__any_sync(0xFFFFFFFFu, any)) break;
            uint64_t cw[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (cas[u]) {
                    cw[u] = atomicCAS(reinterpret_cast<unsigned long long*>(t.slots + hidx(key[u], t.seed[at[u]], t.nslots)),
                                      kEmpty, K::word(key[u], VALUES ? vals[(r * kU + u) * stride + tid] : 0u));
                    ++direct;
                }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (!cas[u]) continue;
                if (cw[u] == kEmpty) {
                    placed[u] = true;
                    cas[u] = false;
                } else if (K::keyof(cw[u]) == key[u]) {
                    cas[u] = false;                        // another copy stored it
                } else if (t.chain_h1 || at[u] + 1 >= t.k) {
                    claim[u] = true;                       // every slot is full now
                    cas[u] = false;
                } else {
                    ++at[u];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint64_t i = (r * kU + u) * stride + tid;
            bool winner = placed[u];
            uint32_t spos = 0;
            if (claim[u]) winner = claim_key<KW>(t, sc, dseed, key[u], &spos);
            if (i < n && out_flag) out_flag[i] = uint8_t(winner);
            stored += placed[u] && !list_stored;
            const bool listed = winner && (list_stored || !placed[u]);
            winners.add(listed, listed ? K::word(key[u], VALUES ? vals[i] : 0u) : 0, i, spos, placed[u]);
        }
    }
    winners.flush();
    add_probe_counters(t, probes, misses, miss_reads, direct, stored);
}

// Lookup: four keys per thread, one slot of each at a time until it is found or
// meets an EMPTY slot.  Without claims to wait for, a queue costs more than the
// lanes it keeps busy: 20 M lookups, half absent, in 8 MB 276 us with the probe
// kernel's queue, 246 here, 32-bit keys with values 380, 265; past L2 at load 0.5
// (2^24 lookups) 662 us, 605 here in 1 GB, 32-bit keys with values 502, 385 in 270
// MB.  Touching the next round's first slots ahead gives nothing (605, 411 us).
// Past L2 bound by random lines.  In L2 2^24 lookups of stored keys (10 MB) take 198
// us, 193 with the kernel before it, which held all k words of a key and is
// slower on others (2^22 32-bit ones 56 us, 51 here; past L2 at load 0.5 446, 433).
template <int KW>
__global__ void __launch_bounds__(kBlock, 3)
cuckoo_lookup_kernel(const __grid_constant__ DevTable t, const void* __restrict__ keys, uint64_t n,
                     uint8_t* __restrict__ found_out, uint32_t* __restrict__ val_out) {
    using K = Keys<KW>;
    pdl_wait();
    const uint32_t stash_used = __ldcg(&t.ctr->stash_used);
    const uint32_t ovf_used = __ldcg(&t.ctr->ovf_used);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t tid = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const uint64_t rounds = (n + stride * kU - 1) / (stride * kU);     // warp-uniform trip count
    unsigned long long probes = 0;
    // The next round's keys are loaded while this round waits on the table.
    uint64_t next_key[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        const uint64_t i = uint64_t(u) * stride + tid;
        next_key[u] = i < n ? K::load(keys, i) : 0;
    }
    for (uint64_t r = 0; r < rounds; ++r) {
        uint64_t key[kU], w[kU];
        bool act[kU], found[kU], more[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint64_t i = (r * kU + u) * stride + tid;
            key[u] = next_key[u];
            const uint64_t j = ((r + 1) * kU + u) * stride + tid;
            if (j < n) next_key[u] = K::load(keys, j);
            act[u] = i < n;
            if (act[u] && K::reserved(key[u])) {
                set_flag(t.ctr, kFlagInvalidKey);
                act[u] = false;
            }
            more[u] = act[u];
            found[u] = false;
            w[u] = kEmpty;
        }
        for (uint32_t a = 0; a < t.k; ++a) {
            bool any = false;
#pragma unroll
            for (int u = 0; u < kU; ++u) any |= more[u];
            if (!__any_sync(0xFFFFFFFFu, any)) break;
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (more[u])
                    w[u] = __ldcg(reinterpret_cast<const unsigned long long*>(t.slots + hidx(key[u], t.seed[a], t.nslots)));
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (!more[u]) continue;
                ++probes;
                found[u] = K::keyof(w[u]) == key[u];
                more[u] = !found[u] && !K::empty(w[u]);
            }
        }
        if (stash_used | ovf_used) {
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (act[u] && !found[u]) found[u] = find_spill<KW>(t, key[u], stash_used, ovf_used, &w[u]);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint64_t i = (r * kU + u) * stride + tid;
            if (i < n) {
                if (found_out) found_out[i] = uint8_t(found[u]);
                if (val_out) val_out[i] = found[u] ? K::value(w[u]) : 0u;
            }
        }
    }
    for (int o = 16; o; o >>= 1) probes += __shfl_down_sync(0xFFFFFFFFu, probes, o);
    unsigned long long* const dst[1] = {&t.ctr->probes};
    const unsigned long long sums[1] = {probes};
    block_add_counters<1>(dst, sums);
}

// Eviction-chain insert of the winners.  Each thread keeps U chains in
// flight so their exchanges overlap, and a chain that ends (an empty slot,
// or the stash) is replaced at once by the thread's next winner: chain
// lengths vary widely at high load, and refilling keeps every slot of the
// thread busy instead of waiting for the longest chain of a round.  Each
// step reads the next records for all free chain slots together with the
// live chains' exchanges.  A record of a key the probe stored (listed only
// for a caller that collects the new keys) holds no claim and is counted.
template <int KW, bool APPEND>
__global__ void __launch_bounds__(kBlock, 3)
cuckoo_insert_kernel(const DevTable t, const DevScratch sc, uint32_t parity, uint64_t max_winners,
                     typename Keys<KW>::T* __restrict__ new_out, unsigned long long* __restrict__ new_count,
                     uint64_t new_cap) {
    using K = Keys<KW>;
    pdl_wait();
    const uint64_t count = min(uint64_t(__ldcg(&t.ctr->winners[parity])), max_winners);
    // The other parity's list was consumed by the previous insert kernel on
    // this stream; reset its counter for the next probe kernel.
    if (blockIdx.x == 0 && threadIdx.x == 0) t.ctr->winners[parity ^ 1u] = 0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t tid = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (APPEND) {
        // Every winner is a new key: append them all, warp-aggregated.
        const uint64_t rounds = (count + stride - 1) / stride;
        for (uint64_t r = 0; r < rounds; ++r) {
            const uint64_t i = r * stride + tid;
            const uint64_t key = i < count ? K::keyof(sc.win[i].word) : 0;
            warp_append<typename K::T>(i < count, typename K::T(key), new_out, new_count, new_cap);
        }
    }
    unsigned long long placed = 0, exchanges = 0;
    uint64_t next = tid;                  // this thread's next winner: tid, tid + stride, ...
    uint64_t word[kU], pos[kU];
    uint32_t evictions[kU];
    bool live[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        live[u] = false;
        word[u] = 0;
        pos[u] = 0;
        evictions[u] = 0;
    }
    // Bounded: each step takes at least one record or runs at least one
    // exchange; each winner is taken once and its chain ends after at most
    // max_evictions + 1 exchanges.
    for (;;) {
        uint32_t nfree = 0;
#pragma unroll
        for (int u = 0; u < kU; ++u) nfree += live[u] ? 0u : 1u;
        Winner rec[kU];
        bool got[kU];
#pragma unroll
        for (int j = 0; j < kU; ++j) {
            got[j] = uint32_t(j) < nfree && next < count;
            if (got[j]) {
                rec[j] = sc.win[next];
                next += stride;
            }
        }
        uint64_t old[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (live[u]) old[u] = atomicExch(reinterpret_cast<unsigned long long*>(t.slots + pos[u]), word[u]);
        bool any = false;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (!live[u]) continue;
            ++exchanges;
            if (K::empty(old[u])) {
                live[u] = false;
                ++placed;
                continue;
            }
            // Section 4.1: the evicted key k' sat at h_a(k') = pos; it moves
            // on to h_{a+1}(k') (cyclically after h_k).
            word[u] = old[u];
            if (++evictions[u] > t.max_evict) {
                // The chain hit the eviction bound: the held word goes to the stash.
                if (place_spill<KW>(t, K::keyof(word[u]), word[u]) == 1) ++placed;
                live[u] = false;
                continue;
            }
            const uint64_t key = K::keyof(old[u]);
            uint32_t a = 0;
            for (; a + 1 < t.k; ++a)
                if (hidx(key, t.seed[a], t.nslots) == pos[u]) break;
            const uint32_t nxt = (a + 1 == t.k) ? 0u : a + 1;
            pos[u] = hidx(key, t.seed[nxt], t.nslots);
            any = true;
        }
        // The records read this step: a key the probe stored is counted; a
        // claimant gives its claim back (the dedup set is left empty for the
        // next batch) and takes a free chain slot (there are at least as
        // many as records read).
#pragma unroll
        for (int j = 0; j < kU; ++j) {
            if (!got[j]) continue;
            if (rec[j].start == kStartPlaced) {
                ++placed;
                continue;
            }
            sc.set[rec[j].spos] = kEmpty;
            bool taken = false;
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (!live[u] && !taken) {
                    word[u] = rec[j].word;
                    pos[u] = hidx(K::keyof(rec[j].word), t.seed[rec[j].start < t.k ? rec[j].start : 0u], t.nslots);
                    evictions[u] = 0;
                    live[u] = true;
                    taken = true;
                }
            any = true;
        }
        if (!any && next >= count) break;
    }
    for (int o = 16; o; o >>= 1) {
        placed += __shfl_down_sync(0xFFFFFFFFu, placed, o);
        exchanges += __shfl_down_sync(0xFFFFFFFFu, exchanges, o);
    }
    unsigned long long* const dst[2] = {&t.ctr->size, &t.ctr->exchanges};
    const unsigned long long sums[2] = {placed, exchanges};
    block_add_counters<2>(dst, sums);
}

}  // namespace

cudaError_t cuckoo_probe(int kw, const DevTable& t, const DevScratch& sc, uint32_t parity,
                         const void* keys, const uint32_t* vals, uint64_t n,
                         const unsigned long long* d_n, uint64_t off, uint8_t* is_new, cudaStream_t s,
                         const L2Window& w, bool list_stored, bool local) {
    ProfScope ps(kKCuckooProbe, s);
    // Tables past L2 with a batch in its own order.  Blocks per SM, 2 / 3: a map of
    // 2^24 keys in 170 MB 1.48 / 1.36 ms, 2^25 keys in 320 MB 3.81 / 3.68; 2^26 in 670
    // MB equal, in 1 GB 5.03 / 5.14, 2^27 in 2.1 GB 10.63 / 10.85.
    const uint64_t bytes = t.nslots * 8, l2 = l2_bytes();
    const bool far = !local && bytes > l2, near = bytes <= 4 * l2;
#define L(KW, V)                                                                                        \
    {                                                                                                   \
        auto k = !far ? cuckoo_probe_kernel<KW, V>                                                      \
                      : near ? cuckoo_probe_far_kernel<KW, V, 3> : cuckoo_probe_far_kernel<KW, V, 2>;   \
        return launch_win(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, w, t, sc, parity, keys, vals, \
                          n, d_n, off, is_new, list_stored);                                            \
    }
    if (kw == 32) {
        if (vals) L(32, true) else L(32, false)
    }
    L(64, false)
#undef L
}

cudaError_t cuckoo_insert(int kw, const DevTable& t, const DevScratch& sc, uint32_t parity,
                          void* new_out, unsigned long long* new_count, uint64_t new_cap,
                          uint64_t max_winners, cudaStream_t s, const L2Window& w) {
    ProfScope ps(kKCuckooInsert, s);
#define L(KW, A)                                                                                        \
    {                                                                                                   \
        auto k = cuckoo_insert_kernel<KW, A>;                                                           \
        return launch_win(k, launch_grid((const void*)k, kBlock, max_winners, kBlock), kBlock, 0, s, w, t, sc, parity, max_winners, \
                          static_cast<typename Keys<KW>::T*>(new_out), new_count, new_cap);             \
    }
    if (kw == 32) {
        if (new_out) L(32, true) else L(32, false)
    }
    if (new_out) L(64, true)
    L(64, false)
#undef L
}

cudaError_t cuckoo_lookup(int kw, const DevTable& t, const void* keys, uint64_t n, uint32_t* vals,
                          uint8_t* found, cudaStream_t s, const L2Window& w) {
    ProfScope ps(kKCuckooLookup, s);
    auto k = kw == 32 ? cuckoo_lookup_kernel<32> : cuckoo_lookup_kernel<64>;
    return launch_win(k, launch_grid((const void*)k, kBlock, n, kBlock), kBlock, 0, s, w, t, keys, n, found, vals);
}

}  // namespace ht
