// csaw_pack.cu -- builds the packed search array of a static bias (PackView):
// the CTPS of Sec. II-B as one running sum over ALL edges, so that rows need
// no segment handling and a row's own sums are differences of it.
//
// One pass over the edges writes the packed groups, their sums inside 64-edge
// blocks and the block ends relative to the thread block's chunk; the chunk
// totals are scanned by one block, then added to the block ends.  Bound by
// memory: 8 bytes read and 8.67 written per edge (neighbour degree adds its
// gathers, once).  RMAT s20, 31 M edges: 0.077 ms for the edges (6.7 TB/s),
// 0.11 in all, against 0.15 for the segmented scan of the summaries.
#include "csaw_internal.cuh"

namespace csaw {

constexpr int PK_THREADS = 256;
constexpr int PK_ROUNDS = (int)(PACK_CHUNK / (8 * PK_THREADS));   // 8-edge groups per thread and chunk

bool pack_fits(const csaw_graph* g, int kind)
{
    // a block's sums in 32 bits, all edges' in 64
    const uint64_t most = kind == CSAW_BIAS_EDGE_WEIGHT ? g->max_weight : g->max_degree;
    if (kind != CSAW_BIAS_EDGE_WEIGHT && kind != CSAW_BIAS_NEIGHBOR_DEGREE) return false;
    if (kind == CSAW_BIAS_EDGE_WEIGHT && !g->w) return false;
    return g->E > 0 && g->E < (1ull << 38) && most < (1ull << 26);
}

template <int KIND>
__global__ void __launch_bounds__(PK_THREADS) pack_groups_kernel(const uint32_t* __restrict__ col,
                                                                 const uint32_t* __restrict__ w,
                                                                 const uint32_t* __restrict__ deg, uint64_t E,
                                                                 uint32_t* __restrict__ pack, uint32_t* __restrict__ s1,
                                                                 uint64_t* __restrict__ s2,
                                                                 uint64_t* __restrict__ chunk_sum)
{
    __shared__ uint64_t s_warp[2][PK_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t running = 0;
    for (int round = 0; round < PK_ROUNDS; ++round) {
        const uint64_t g = (uint64_t)blockIdx.x * (PACK_CHUNK / 8) + (uint64_t)round * PK_THREADS + threadIdx.x;
        const uint64_t e = 8 * g;
        uint32_t c[8] = {0, 0, 0, 0, 0, 0, 0, 0}, b[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (e < E) {   // the arrays' padding covers the last group
            const uint4 c0 = __ldcs(reinterpret_cast<const uint4*>(col + e));
            const uint4 c1 = __ldcs(reinterpret_cast<const uint4*>(col + e) + 1);
            c[0] = c0.x; c[1] = c0.y; c[2] = c0.z; c[3] = c0.w;
            c[4] = c1.x; c[5] = c1.y; c[6] = c1.z; c[7] = c1.w;
            if constexpr (KIND == CSAW_BIAS_EDGE_WEIGHT) {
                const uint4 w0 = __ldcs(reinterpret_cast<const uint4*>(w + e));
                const uint4 w1 = __ldcs(reinterpret_cast<const uint4*>(w + e) + 1);
                b[0] = w0.x; b[1] = w0.y; b[2] = w0.z; b[3] = w0.w;
                b[4] = w1.x; b[5] = w1.y; b[6] = w1.z; b[7] = w1.w;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) b[j] = __ldg(deg + c[j]);
            }
            if (e + 8 > E) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (e + j >= E) b[j] = 0u;
            }
        }
        st256_stream(pack + 16 * g, b);
        st256_stream(pack + 16 * g + 8, c);
        uint32_t in_block = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) in_block += b[j];
        const uint32_t mine = in_block;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const uint32_t y = __shfl_up_sync(CSAW_FULL_MASK, in_block, o, 8);
            if ((lane & 7) >= o) in_block += y;
        }
        s1[g] = in_block;
        const uint64_t incl = warp_inclusive_scan_u64(mine, lane);
        uint64_t* sw = s_warp[round & 1];
        if (lane == 31) sw[wid] = incl;
        __syncthreads();
        uint64_t before = running;
#pragma unroll
        for (int k = 0; k < PK_THREADS / 32; ++k) {
            const uint64_t t = sw[k];
            if (k < wid) before += t;
            running += t;
        }
        if ((lane & 7) == 7) s2[pack_before((uint32_t)(g >> 3)) + 1] = before + incl;
    }
    if (threadIdx.x == 0) chunk_sum[blockIdx.x] = running;
}

// One block: chunk_sum becomes the sum before each chunk.
__global__ void __launch_bounds__(1024) pack_carry_kernel(uint64_t* __restrict__ chunk_sum, uint64_t n)
{
    __shared__ uint64_t s_warp[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t per = (n + 1023) / 1024;
    const uint64_t t0 = min(per * threadIdx.x, n), t1 = min(t0 + per, n);
    uint64_t mine = 0;
    for (uint64_t t = t0; t < t1; ++t) mine += chunk_sum[t];
    const uint64_t incl = warp_inclusive_scan_u64(mine, lane);
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    uint64_t acc = incl - mine;
    for (int k = 0; k < wid; ++k) acc += s_warp[k];
    for (uint64_t t = t0; t < t1; ++t) {
        const uint64_t here = chunk_sum[t];
        chunk_sum[t] = acc;
        acc += here;
    }
}

// The blocks' ends from all edges; a window's first word is the end before it.
__global__ void pack_ends_kernel(const uint64_t* __restrict__ chunk_sum, uint64_t blocks, uint64_t* __restrict__ s2)
{
    for (uint64_t h = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; h < blocks; h += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t at = pack_before((uint32_t)h) + 1;
        const uint64_t end = s2[at] + __ldg(chunk_sum + h / (PACK_CHUNK / 64));
        s2[at] = end;
        if (h % 3 == 2) s2[at + 1] = end;
        if (h == 0) s2[0] = 0;
        if (h + 1 == blocks)
            for (uint64_t q = at + (h % 3 == 2 ? 2 : 1); q < 4 * (blocks / 3 + 1); ++q) s2[q] = ~0ull;
    }
}

// rec[v] = {off[v], the sum of all edges before it}, v <= V.
__global__ void pack_rows_kernel(const uint64_t* __restrict__ off, uint32_t V, const uint32_t* __restrict__ pack,
                                 const uint32_t* __restrict__ s1, const uint64_t* __restrict__ s2,
                                 uint64_t* __restrict__ rec)
{
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= V; v += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t e = __ldg(off + v), g = e >> 3;
        uint64_t before = s2[pack_before((uint32_t)(g >> 3))];
        if (g & 7) before += s1[g - 1];
        for (uint32_t j = 0; j < (uint32_t)(e & 7); ++j) before += pack[16 * g + j];
        reinterpret_cast<ulonglong2*>(rec)[v] = make_ulonglong2(e, before);
    }
}

csaw_status enqueue_pack_build(const csaw_graph* g, int kind, uint64_t* words, cudaStream_t s)
{
    const PackLayout L = pack_layout(g->E, g->V);
    uint32_t* pack = (uint32_t*)words;
    uint32_t* s1 = (uint32_t*)(words + L.s1);
    uint64_t* s2 = words + L.s2;
    uint64_t* rec = words + L.rec;
    uint64_t* cs = words + L.sums;
    if (kind == CSAW_BIAS_EDGE_WEIGHT)
        pack_groups_kernel<CSAW_BIAS_EDGE_WEIGHT><<<(unsigned)L.chunks, PK_THREADS, 0, s>>>(g->col, g->w, g->deg, g->E,
                                                                                            pack, s1, s2, cs);
    else
        pack_groups_kernel<CSAW_BIAS_NEIGHBOR_DEGREE><<<(unsigned)L.chunks, PK_THREADS, 0, s>>>(g->col, g->w, g->deg,
                                                                                                g->E, pack, s1, s2, cs);
    pack_carry_kernel<<<1, 1024, 0, s>>>(cs, L.chunks);
    const auto grid = [&](uint64_t n) {
        const uint64_t b = (n + 255) / 256, cap = (uint64_t)g->sm_count * 16;
        return (unsigned)(b < cap ? b : cap);
    };
    pack_ends_kernel<<<grid(L.blocks), 256, 0, s>>>(cs, L.blocks, s2);
    pack_rows_kernel<<<grid((uint64_t)g->V + 1), 256, 0, s>>>(g->off, g->V, pack, s1, s2, rec);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? CSAW_OK : cuda_fail(e, "packed array launch");
}

}  // namespace csaw
