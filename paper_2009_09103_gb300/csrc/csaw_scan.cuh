// csaw_scan.cuh -- block-wide pieces of the device-wide scan and of the
// frontier construction that is fused with it.
#pragma once

#include "csaw_internal.cuh"

namespace csaw {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr uint64_t SCAN_TILE = (uint64_t)SCAN_THREADS * SCAN_ITEMS;
constexpr int SCAN_MAX_BLOCKS = 1024;

// Blocks of a scan of up to n_max elements (csaw_prims.cu).
int scan_blocks(uint64_t n_max);

// The contiguous range of tiles that this block owns.
__device__ __forceinline__ void block_range(uint64_t n, uint64_t tile, uint64_t* lo, uint64_t* hi)
{
    const uint64_t tiles = (n + tile - 1) / tile;
    const uint64_t per = (tiles + gridDim.x - 1) / gridDim.x;
    uint64_t b = (uint64_t)blockIdx.x * per * tile;
    uint64_t e = b + per * tile;
    *lo = b < n ? b : n;
    *hi = e < n ? e : n;
}

// Block-wide exclusive scan of one uint64 per thread; returns the block total.
__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t* excl, uint64_t* s_warp)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t incl = warp_inclusive_scan_u64(v, lane);
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int nw = blockDim.x >> 5;
        uint64_t t = lane < nw ? s_warp[lane] : 0;
        const uint64_t ti = warp_inclusive_scan_u64(t, lane);
        if (lane < nw) s_warp[lane] = ti - t;
        if (lane == nw - 1) s_warp[32] = ti;
    }
    __syncthreads();
    *excl = s_warp[wid] + incl - v;
    const uint64_t total = s_warp[32];
    __syncthreads();
    return total;
}

// The sum of the first n block totals.
__device__ __forceinline__ uint64_t sum_before(const uint64_t* __restrict__ bsum, uint32_t n, uint64_t* s_warp)
{
    uint64_t t = 0, excl;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) t += bsum[i];
    return block_exclusive_scan(t, &excl, s_warp);
}

// out[i] = base + in[t0] + ... + in[i - 1] over the tile [t0, min(t0 + SCAN_TILE, hi));
// returns the tile's total.
__device__ __forceinline__ uint64_t scan_tile(const uint32_t* __restrict__ in, uint64_t t0, uint64_t hi,
                                              uint64_t base, uint64_t* __restrict__ out, uint64_t* s_warp)
{
    const uint64_t my = t0 + (uint64_t)threadIdx.x * SCAN_ITEMS;
    uint32_t v[SCAN_ITEMS];
    uint64_t s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        v[j] = (my + j < hi) ? in[my + j] : 0u;
        s += v[j];
    }
    uint64_t excl;
    const uint64_t total = block_exclusive_scan(s, &excl, s_warp);
    uint64_t run = base + excl;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        if (my + j < hi) out[my + j] = run;
        run += v[j];
    }
    return total;
}

}  // namespace csaw
