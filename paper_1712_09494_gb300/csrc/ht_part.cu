// Reordering a large batch by the table region its keys' first bucket (slot)
// lies in, so that find-or-put works on one L2-sized region of a table larger
// than L2 after another (ht_api.cu decides when).
//
// Random lines of a large table come from DRAM at 40-46 G lines/s, 25 G/s where
// they are also written.  A batch with more than one key per 128-byte line of
// the table touches many lines twice or more; taken region by region each line
// is fetched and written back once, and the probes and claims run in L2.
// Two passes over the keys: count per region, then move; and one over the
// answers, which the table's kernels write in region order, back to the batch's.
// Bound by their bytes: 8 read, 8 read and 10 written, 3 read and 1 written per
// 64-bit key (2^24 keys: 28, 80 and 25 us).
#include <algorithm>

#include "ht_internal.cuh"

namespace ht {
namespace {

constexpr int kPartThreads = 512;
constexpr int kPartPer = int(kPartTile) / kPartThreads;   // keys per thread

// The region of a key: the top bits of its first hash, which the range
// reduction to a bucket or slot keeps in order.
__device__ __forceinline__ uint32_t region_of(uint64_t key, uint64_t seed, int shift) {
    return uint32_t(mix64(key ^ seed) >> shift);
}
__device__ __forceinline__ uint32_t region_of(const ulonglong2& key, uint64_t seed, int shift) {
    return region_of(wide_fold(key.x, key.y), seed, shift);
}

template <typename T>
__global__ void __launch_bounds__(kPartThreads)
part_count_kernel(const T* __restrict__ keys, uint64_t n, const unsigned long long* __restrict__ d_n, uint64_t seed,
                  int shift, unsigned int* __restrict__ hist) {
    __shared__ unsigned int s_cnt[kMaxRegions];
    pdl_wait();
    if (d_n) n = min(n, uint64_t(__ldcg(d_n)));
    for (int i = threadIdx.x; i < kMaxRegions; i += kPartThreads) s_cnt[i] = 0;
    __syncthreads();
    const uint64_t stride = uint64_t(gridDim.x) * kPartThreads;
    uint64_t i = uint64_t(blockIdx.x) * kPartThreads + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {         // four loads in flight
        T k[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) k[j] = keys[i + j * stride];
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicAdd(&s_cnt[region_of(k[j], seed, shift)], 1u);
    }
    for (; i < n; i += stride) atomicAdd(&s_cnt[region_of(keys[i], seed, shift)], 1u);
    __syncthreads();
    for (int r = threadIdx.x; r < kMaxRegions; r += kPartThreads)
        if (s_cnt[r]) atomicAdd(hist + r, s_cnt[r]);
}

// A block takes 4096 keys, sorts them by region in shared memory and writes each
// region's run to its place, reserved with one atomic per block and region.
// BACK: with each key's place in its tile, and the tile's runs (start and length
// per region), for part_back_kernel.
template <typename T, bool BACK>
__global__ void __launch_bounds__(kPartThreads, sizeof(T) > 8 ? 2 : 3)
part_move_kernel(const T* __restrict__ keys, uint64_t n, const unsigned long long* __restrict__ d_n, uint64_t seed,
                 int shift, const unsigned int* __restrict__ hist, unsigned int* __restrict__ cursor,
                 T* __restrict__ out, uint16_t* __restrict__ loc, uint2* __restrict__ runs) {
    extern __shared__ __align__(16) unsigned char smem[];
    T* s_key = reinterpret_cast<T*>(smem);
    uint8_t* s_reg = reinterpret_cast<uint8_t*>(s_key + kPartTile);
    uint16_t* s_loc = reinterpret_cast<uint16_t*>(s_reg + kPartTile);
    const uint32_t regions = 1u << (64 - shift);
    __shared__ unsigned int s_cnt[kMaxRegions];           // keys of the tile per region
    __shared__ unsigned int s_start[kMaxRegions];         // their start in the sorted tile
    __shared__ unsigned int s_first[kMaxRegions];         // the region's start in out
    __shared__ unsigned int s_at[kMaxRegions];            // this tile's run in out
    __shared__ unsigned int s_warp[kMaxRegions / 32];
    pdl_wait();
    if (d_n) n = min(n, uint64_t(__ldcg(d_n)));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Exclusive scan of one value per region (threads < kMaxRegions).
    auto scan = [&](unsigned int v) {
        unsigned int incl = v;
        if (tid < kMaxRegions) {
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int x = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += x;
            }
            if (lane == 31) s_warp[warp] = incl;
        }
        __syncthreads();
        unsigned int before = 0;
        if (tid < kMaxRegions)
            for (int w = 0; w < warp; ++w) before += s_warp[w];
        __syncthreads();
        return before + incl - v;
    };
    static_assert(kMaxRegions <= kPartThreads && kMaxRegions % 32 == 0, "one thread per region");
    const unsigned int first = scan(tid < kMaxRegions ? hist[tid] : 0u);
    if (tid < kMaxRegions) s_first[tid] = first;
    for (uint64_t base = uint64_t(blockIdx.x) * kPartTile; base < n; base += uint64_t(gridDim.x) * kPartTile) {
        if (tid < kMaxRegions) s_cnt[tid] = 0;
        __syncthreads();
        T key[kPartPer];
        uint32_t at[kPartPer];                            // region << 16 | rank in it
#pragma unroll
        for (int j = 0; j < kPartPer; ++j) {
            const uint64_t i = base + uint32_t(j * kPartThreads + tid);
            key[j] = i < n ? keys[i] : T{};
        }
#pragma unroll
        for (int j = 0; j < kPartPer; ++j) {
            const uint64_t i = base + uint32_t(j * kPartThreads + tid);
            const uint32_t r = region_of(key[j], seed, shift);
            at[j] = i < n ? (r << 16) | atomicAdd(&s_cnt[r], 1u) : ~0u;
        }
        __syncthreads();
        const unsigned int c = tid < kMaxRegions ? s_cnt[tid] : 0u;
        const unsigned int st = scan(c);
        if (tid < kMaxRegions) {
            s_start[tid] = st;
            const unsigned int o = s_first[tid] + (c ? atomicAdd(cursor + tid, c) : 0u);
            s_at[tid] = o - st;
            if (BACK && tid < regions) runs[base / kPartTile * regions + tid] = make_uint2(o, c);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPartPer; ++j)
            if (at[j] != ~0u) {
                const uint32_t p = s_start[at[j] >> 16] + (at[j] & 0xFFFFu);
                s_key[p] = key[j];
                s_reg[p] = uint8_t(at[j] >> 16);
                if (BACK) s_loc[p] = uint16_t(j * kPartThreads + tid);
            }
        __syncthreads();
        const uint32_t m = uint32_t(min(uint64_t(kPartTile), n - base));
        for (uint32_t p = tid; p < m; p += kPartThreads) {
            const uint32_t o = s_at[s_reg[p]] + p;
            out[o] = s_key[p];
            if (BACK) loc[o] = s_loc[p];
        }
        __syncthreads();
    }
}

// The answers of a tile's keys, from region order back to the batch's: a warp
// per run, through shared memory, so that both sides are read and written in
// runs (written straight from the table's kernels, one byte at a random place
// each, they cost 110 us per 2^24 keys; this pass takes 25).
__global__ void __launch_bounds__(kPartThreads)
part_back_kernel(const uint8_t* __restrict__ from, const uint16_t* __restrict__ loc, const uint2* __restrict__ runs,
                 uint32_t regions, uint64_t n, uint8_t* __restrict__ to) {
    __shared__ __align__(16) uint8_t s_out[kPartTile];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait();
    for (uint64_t base = uint64_t(blockIdx.x) * kPartTile; base < n; base += uint64_t(gridDim.x) * kPartTile) {
        for (uint32_t r = warp; r < regions; r += kPartThreads / 32) {
            const uint2 run = runs[base / kPartTile * regions + r];
            for (uint32_t j = lane; j < run.y; j += 32) s_out[loc[run.x + j]] = from[run.x + j];
        }
        __syncthreads();
        const uint32_t m = uint32_t(min(uint64_t(kPartTile), n - base));
        uint8_t* o = to + base;
        if (m == kPartTile && (reinterpret_cast<uintptr_t>(o) & 15) == 0) {
            for (uint32_t p = threadIdx.x; p < kPartTile / 16; p += kPartThreads)
                reinterpret_cast<uint4*>(o)[p] = reinterpret_cast<const uint4*>(s_out)[p];
        } else {
            for (uint32_t p = threadIdx.x; p < m; p += kPartThreads) o[p] = s_out[p];
        }
        __syncthreads();
    }
}

template <typename T>
cudaError_t part_run(const T* keys, uint64_t n, const unsigned long long* d_n, uint64_t seed, int bits, unsigned int* ctl,
                     T* out, uint16_t* loc, uint2* runs, cudaStream_t s) {
    const int shift = 64 - bits;
    cudaError_t e = cudaMemsetAsync(ctl, 0, 2 * kMaxRegions * sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    auto c = part_count_kernel<T>;
    e = launch_after(c, launch_grid((const void*)c, kPartThreads, n, kPartTile), kPartThreads, 0, s, keys, n, d_n, seed,
                     shift, ctl);
    if (e != cudaSuccess) return e;
    auto k = loc ? part_move_kernel<T, true> : part_move_kernel<T, false>;
    const size_t smem = kPartTile * (sizeof(T) + 1 + (loc ? 2 : 0));
    e = allow_smem((const void*)k, smem);
    if (e != cudaSuccess) return e;
    return launch_after(k, launch_grid((const void*)k, kPartThreads, n, kPartTile, smem), kPartThreads, smem, s, keys, n,
                        d_n, seed, shift, ctl, ctl + kMaxRegions, out, loc, runs);
}

}  // namespace

cudaError_t partition_keys(int kw, const void* keys, uint64_t n, const unsigned long long* d_n, uint64_t seed, int bits,
                           unsigned int* ctl, void* out, uint16_t* loc, void* runs, cudaStream_t s) {
    ProfScope ps(kKPartition, s);
    uint2* r = static_cast<uint2*>(runs);
    if (kw == 32)
        return part_run(static_cast<const uint32_t*>(keys), n, d_n, seed, bits, ctl, static_cast<uint32_t*>(out), loc, r, s);
    if (kw == 128)
        return part_run(static_cast<const ulonglong2*>(keys), n, d_n, seed, bits, ctl, static_cast<ulonglong2*>(out), loc,
                        r, s);
    return part_run(static_cast<const uint64_t*>(keys), n, d_n, seed, bits, ctl, static_cast<uint64_t*>(out), loc, r, s);
}

cudaError_t partition_back(const uint8_t* from, const uint16_t* loc, const void* runs, int bits, uint64_t n, uint8_t* to,
                           cudaStream_t s) {
    ProfScope ps(kKPartition, s);
    auto k = part_back_kernel;
    return launch_after(k, launch_grid((const void*)k, kPartThreads, n, kPartTile), kPartThreads, 0, s, from, loc,
                        static_cast<const uint2*>(runs), 1u << bits, n, to);
}

}  // namespace ht
