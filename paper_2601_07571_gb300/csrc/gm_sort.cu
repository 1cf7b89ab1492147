// gm_sort.cu -- stable LSD radix sort (8-bit digits) and an int64 inclusive scan.
//
// Used by the BVH build (Morton keys of triangle centroids), the spatial work order of the
// samples, the window sort of fixations, and the fixed-point prefix of per-triangle counts.
// Up to RS_SMALL keys: one block sorts them in shared memory, one launch for all digits. More: three
// kernels per radix pass: per-tile digit histograms, an exclusive scan of every digit's row of the
// digit-major histogram table (a block per digit), then a stable scatter in which each warp ranks its
// own run of keys with warp match and its own digit counters, so that a tile synchronises five times (three
// of them the scan's) rather than three times per 256 keys. Tiles of 2048 keys: at 800k keys they make 390 blocks (196 of
// 4096 keys left the 152 SMs at one block each). No spin-waits anywhere.
// Bound by launches and latency at these sizes (800k 63-bit keys: 19 MB a pass).
#include <algorithm>

#include "gm_blocksort.cuh"
#include "gm_internal.cuh"
#include "gm_scan.cuh"

namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;
constexpr int RS_WARPS = RS_THREADS / 32;

template <typename K>
__global__ void __launch_bounds__(RS_THREADS) rs_hist(const K* __restrict__ keys, uint32_t n, int shift,
                                                      uint32_t* __restrict__ hist, uint32_t nblocks) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t base = blockIdx.x * (uint32_t)RS_TILE;
    uint32_t d[RS_ITEMS];
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const uint32_t idx = base + i * RS_THREADS + threadIdx.x;
        d[i] = idx < n ? (uint32_t)((keys[idx] >> shift) & 255u) : 256u;
    }
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const unsigned peers = __match_any_sync(0xffffffffu, d[i]);
        if (d[i] < 256u && (peers & gm_lanemask_lt()) == 0) atomicAdd(&h[d[i]], (uint32_t)__popc(peers));
    }
    __syncthreads();
    hist[(size_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Block d: exclusive scan of digit d's counts over the tiles, in place, and their total.
__global__ void __launch_bounds__(RS_THREADS) rs_scan(uint32_t* __restrict__ hist, uint32_t nblocks,
                                                      uint32_t* __restrict__ totals) {
    uint32_t* a = hist + (size_t)blockIdx.x * nblocks;
    uint32_t carry = 0;
    for (uint32_t base = 0; base < nblocks; base += RS_THREADS) {
        const uint32_t i = base + threadIdx.x;
        const uint32_t v = i < nblocks ? a[i] : 0u;
        uint32_t tot;
        const uint32_t ex = block_excl_scan<uint32_t, RS_THREADS>(v, &tot);
        if (i < nblocks) a[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// Rank of each lane's digit among the warp's equal digits so far (stable in lane order), counting
// them in the warp's own counters. d = 256: no key.
__device__ __forceinline__ uint32_t rs_warp_rank(uint32_t d, uint32_t* counters) {
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const uint32_t before = d < 256u ? counters[d] : 0u;
    __syncwarp();
    if (d < 256u && (peers & gm_lanemask_lt()) == 0) counters[d] = before + __popc(peers);
    __syncwarp();
    return before + __popc(peers & gm_lanemask_lt());
}

template <typename K>
__global__ void __launch_bounds__(RS_THREADS) rs_scatter(const K* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                         K* __restrict__ kout, uint32_t* __restrict__ vout,
                                                         uint32_t n, int shift, const uint32_t* __restrict__ hist,
                                                         uint32_t nblocks, const uint32_t* __restrict__ totals) {
    __shared__ uint32_t dbase[256];
    __shared__ uint32_t wcount[RS_WARPS][256];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) wcount[w][tid] = 0;
    // a warp takes RS_ITEMS x 32 consecutive keys
    const uint32_t base = blockIdx.x * (uint32_t)RS_TILE + warp * (32 * RS_ITEMS) + lane;
    K k[RS_ITEMS];
    uint32_t v[RS_ITEMS], rank[RS_ITEMS];
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const uint32_t idx = base + i * 32;
        k[i] = idx < n ? kin[idx] : K(0);
        v[i] = idx < n ? vin[idx] : 0u;
    }
    uint32_t all;
    const uint32_t below = block_excl_scan<uint32_t, RS_THREADS>(totals[tid], &all);   // (synchronises)
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i)
        rank[i] = rs_warp_rank(base + i * 32 < n ? (uint32_t)((k[i] >> shift) & 255u) : 256u, wcount[warp]);
    __syncthreads();
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {
        const uint32_t c = wcount[w][tid];
        wcount[w][tid] = run;
        run += c;
    }
    dbase[tid] = below + hist[(size_t)tid * nblocks + blockIdx.x];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        if (base + i * 32 >= n) continue;
        const uint32_t d = (uint32_t)((k[i] >> shift) & 255u);
        const uint32_t pos = dbase[d] + wcount[warp][d] + rank[i];
        kout[pos] = k[i];
        vout[pos] = v[i];
    }
}

// All passes of n <= RS_SMALL keys in one block, in place.
template <typename K>
__global__ void __launch_bounds__(1024) rs_small(K* __restrict__ keys, uint32_t* __restrict__ vals, uint32_t n, int bits) {
    __shared__ BlockSort<K> B;
    const uint32_t base = block_sort_base();
    K k[RS_PER];
    uint32_t v[RS_PER];
#pragma unroll
    for (int i = 0; i < RS_PER; ++i) {
        const uint32_t idx = base + i * 32;
        k[i] = idx < n ? keys[idx] : K(0);
        v[i] = idx < n ? vals[idx] : 0u;
    }
    block_sort(k, v, n, bits, B);
#pragma unroll
    for (int i = 0; i < RS_PER; ++i) {
        const uint32_t idx = base + i * 32;
        if (idx < n) {
            keys[idx] = k[i];
            vals[idx] = v[i];
        }
    }
}

// The passes proper, with caller-provided temporaries (n keys, n values, 256 * (tiles + 1) counters).
template <typename K>
cudaError_t radix_passes(K* keys, uint32_t* vals, uint32_t n, int bits, K* k2, uint32_t* v2, uint32_t* hist,
                         cudaStream_t s, int* launches) {
    if (n <= 1 || bits <= 0) return cudaSuccess;
    if (n <= RS_SMALL) {
        rs_small<K><<<1, 1024, 0, s>>>(keys, vals, n, bits);
        if (launches) *launches += 1;
        return cudaGetLastError();
    }
    const uint32_t nb = gm_div_up(n, RS_TILE);
    uint32_t* totals = hist + 256 * (size_t)nb;
    K *ka = keys, *kb = k2;
    uint32_t *va = vals, *vb = v2;
    int passes = 0;
    for (int shift = 0; shift < bits; shift += 8, ++passes) {
        rs_hist<K><<<nb, RS_THREADS, 0, s>>>(ka, n, shift, hist, nb);
        rs_scan<<<256, RS_THREADS, 0, s>>>(hist, nb, totals);
        rs_scatter<K><<<nb, RS_THREADS, 0, s>>>(ka, va, kb, vb, n, shift, hist, nb, totals);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    if (launches) *launches += 3 * passes;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && ka != keys) {
        e = cudaMemcpyAsync(keys, ka, sizeof(K) * n, cudaMemcpyDeviceToDevice, s);
        if (e == cudaSuccess) e = cudaMemcpyAsync(vals, va, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, s);
    }
    return e;
}

template <typename K>
gm_status radix_sort(K* keys, uint32_t* vals, uint32_t n, int bits, cudaStream_t s, int* launches) {
    if (n <= 1 || bits <= 0) return GM_OK;
    if (n <= RS_SMALL) {   // one block, no temporaries
        const cudaError_t e = radix_passes<K>(keys, vals, n, bits, nullptr, nullptr, nullptr, s, launches);
        return e == cudaSuccess ? GM_OK : gm_cuda_error(e, "radix sort");
    }
    const uint32_t nb = gm_div_up(n, RS_TILE);
    K* k2 = nullptr;
    uint32_t *v2 = nullptr, *hist = nullptr;
    gm_status st = gm_alloc((void**)&k2, sizeof(K) * n, s);
    if (st == GM_OK) st = gm_alloc((void**)&v2, sizeof(uint32_t) * n, s);
    if (st == GM_OK) st = gm_alloc((void**)&hist, sizeof(uint32_t) * 256 * ((size_t)nb + 1), s);
    if (st != GM_OK) {
        if (k2) cudaFreeAsync(k2, s);
        if (v2) cudaFreeAsync(v2, s);
        return st;
    }
    cudaError_t e = radix_passes<K>(keys, vals, n, bits, k2, v2, hist, s, launches);
    cudaFreeAsync(k2, s);
    cudaFreeAsync(v2, s);
    cudaFreeAsync(hist, s);
    if (e != cudaSuccess) return gm_cuda_error(e, "radix sort");
    return GM_OK;
}

// ---- int64 inclusive scan: tile reduce, scan of tile sums, tile scan + offset ----------------
constexpr int SC_THREADS = 256;
constexpr int SC_ITEMS = 8;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;

__global__ void __launch_bounds__(SC_THREADS) scan_reduce(const int64_t* __restrict__ a, uint32_t n,
                                                          int64_t* __restrict__ part) {
    const uint32_t base = blockIdx.x * (uint32_t)SC_TILE;
    int64_t s = 0;
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        uint32_t idx = base + i * SC_THREADS + threadIdx.x;
        if (idx < n) s += a[idx];
    }
    int64_t tot;
    block_excl_scan<int64_t, SC_THREADS>(s, &tot);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) scan_parts(int64_t* __restrict__ part, uint32_t nb) {
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint32_t base = 0; base < nb; base += 1024) {
        uint32_t i = base + threadIdx.x;
        int64_t v = i < nb ? part[i] : 0;
        int64_t tot;
        int64_t ex = block_excl_scan<int64_t, 1024>(v, &tot);
        if (i < nb) part[i] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(SC_THREADS) scan_down(int64_t* __restrict__ a, uint32_t n,
                                                        const int64_t* __restrict__ part) {
    __shared__ int64_t tile[SC_TILE];
    const uint32_t base = blockIdx.x * (uint32_t)SC_TILE;
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        uint32_t idx = base + i * SC_THREADS + threadIdx.x;
        tile[i * SC_THREADS + threadIdx.x] = idx < n ? a[idx] : 0;
    }
    __syncthreads();
    int64_t v[SC_ITEMS], s = 0;
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        v[i] = tile[threadIdx.x * SC_ITEMS + i];
        s += v[i];
        v[i] = s;
    }
    int64_t tot;
    int64_t ex = block_excl_scan<int64_t, SC_THREADS>(s, &tot) + part[blockIdx.x];
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) tile[threadIdx.x * SC_ITEMS + i] = v[i] + ex;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SC_ITEMS; ++i) {
        uint32_t idx = base + i * SC_THREADS + threadIdx.x;
        if (idx < n) a[idx] = tile[i * SC_THREADS + threadIdx.x];
    }
}

}  // namespace

gm_status gm_radix_sort_u64(uint64_t* keys, uint32_t* vals, uint32_t n, int bits, cudaStream_t s, int* launches) {
    return radix_sort<uint64_t>(keys, vals, n, bits, s, launches);
}

gm_status gm_radix_sort_u32(uint32_t* keys, uint32_t* vals, uint32_t n, int bits, cudaStream_t s, int* launches) {
    return radix_sort<uint32_t>(keys, vals, n, std::min(bits, 32), s, launches);
}

size_t gm_radix_sort_u32_hist_words(uint32_t n) { return 256 * ((size_t)gm_div_up(n, RS_TILE) + 1); }

gm_status gm_radix_sort_u32_prealloc(uint32_t* keys, uint32_t* vals, uint32_t n, int bits, uint32_t* tmp_keys,
                                     uint32_t* tmp_vals, uint32_t* hist, cudaStream_t s, int* launches) {
    cudaError_t e = radix_passes<uint32_t>(keys, vals, n, std::min(bits, 32), tmp_keys, tmp_vals, hist, s, launches);
    if (e != cudaSuccess) return gm_cuda_error(e, "radix sort");
    return GM_OK;
}

gm_status gm_inclusive_scan_i64(int64_t* data, uint32_t n, cudaStream_t s, int* launches) {
    if (n == 0) return GM_OK;
    const uint32_t nb = gm_div_up(n, SC_TILE);
    int64_t* part = nullptr;
    GM_TRY(gm_alloc((void**)&part, sizeof(int64_t) * nb, s));
    scan_reduce<<<nb, SC_THREADS, 0, s>>>(data, n, part);
    scan_parts<<<1, 1024, 0, s>>>(part, nb);
    scan_down<<<nb, SC_THREADS, 0, s>>>(data, n, part);
    if (launches) *launches += 3;
    cudaError_t e = cudaGetLastError();
    cudaFreeAsync(part, s);
    if (e != cudaSuccess) return gm_cuda_error(e, "int64 scan");
    return GM_OK;
}
