// gm_blocksort.cuh -- stable radix sort of up to RS_SMALL (key, value) pairs held by one block of 1024
// threads, all digits in one go: each warp ranks its own run of keys with warp match and its own digit
// counters.
#pragma once

#include "gm_internal.cuh"
#include "gm_scan.cuh"

namespace {

constexpr int RS_SMALL = 2048;
constexpr int RS_PER = RS_SMALL / 1024;   // pairs a thread

template <typename K>
struct BlockSort {
    K key[RS_SMALL];
    uint32_t val[RS_SMALL];
    uint16_t count[32][256];
    uint32_t base[256];
};

// A thread's pair i stands at block_sort_base() + 32 i.
__device__ __forceinline__ uint32_t block_sort_base() {
    return (threadIdx.x >> 5) * (32 * RS_PER) + (threadIdx.x & 31);
}

// Sorts the n pairs by the low `bits` bits of the keys. All threads of a block of 1024 call it.
template <typename K>
__device__ __forceinline__ void block_sort(K (&k)[RS_PER], uint32_t (&v)[RS_PER], uint32_t n, int bits, BlockSort<K>& B) {
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t base = block_sort_base();
    for (int shift = 0; shift < bits; shift += 8) {
        for (int i = tid; i < 32 * 256; i += 1024) (&B.count[0][0])[i] = 0;
        __syncthreads();
        uint32_t rank[RS_PER];
#pragma unroll
        for (int i = 0; i < RS_PER; ++i) {
            const uint32_t d = base + i * 32 < n ? (uint32_t)((k[i] >> shift) & 255u) : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const uint32_t before = d < 256u ? B.count[warp][d] : 0u;
            __syncwarp();
            if (d < 256u && (peers & gm_lanemask_lt()) == 0) B.count[warp][d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            rank[i] = before + __popc(peers & gm_lanemask_lt());
        }
        __syncthreads();
        uint32_t run = 0;
        if (tid < 256) {
            for (int w = 0; w < 32; ++w) {
                const uint32_t c = B.count[w][tid];
                B.count[w][tid] = (uint16_t)run;
                run += c;
            }
        }
        uint32_t all;
        const uint32_t below = block_excl_scan<uint32_t, 1024>(run, &all);
        if (tid < 256) B.base[tid] = below;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RS_PER; ++i) {
            if (base + i * 32 >= n) continue;
            const uint32_t d = (uint32_t)((k[i] >> shift) & 255u);
            const uint32_t pos = B.base[d] + B.count[warp][d] + rank[i];
            B.key[pos] = k[i];
            B.val[pos] = v[i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RS_PER; ++i) {
            const uint32_t idx = base + i * 32;
            if (idx < n) {
                k[i] = B.key[idx];
                v[i] = B.val[idx];
            }
        }
    }
}

}  // namespace
