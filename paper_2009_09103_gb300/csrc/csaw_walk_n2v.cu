// csaw_walk_n2v.cu -- node2vec walks by intersection of neighbour lists
// (Sec. II-A; dynamic bias), one warp per walker.
//
// The biases of a node2vec step at cur, entered from prev, are w * m2 but for
// the common neighbours J of the two vertices (w * m1) and prev itself
// (w * m0).  Which neighbours are common is found from the SHORTER of the two
// lists: its ids are looked up in the longer one, so that a step costs
// min(d_cur, d_prev) look-ups instead of a pass over d_cur (685 against 3,315
// on average on RMAT s20 ef32, where walks live on hubs).  Two forms:
//   list = N(cur):  every bias of the row is formed while its ids are looked
//                   up in N(prev); the pick is a prefix-sum search over them.
//   list = N(prev): only J's weights are summed; with W the row's weight
//                   prefix sums (summaries built for the call, w_search),
//                     S[i] = m2*W[i] + (m1-m2)*sum_{j in J, j<=i} w_j
//                            + (m0-m2)*w_p*[p <= i]
//                   (p the position of prev), in wrapping 64-bit arithmetic,
//                   exact because every true value fits.
// Both give the integers of the streaming kernel (walk_kernel<NODE2VEC>), so
// the paths are the same.
//
// Look-up: a per-call index cuts every row's id span into ranges (8 to 16 per
// neighbour), one bit each, in words of 32 beside the number of the row's ids
// before the word.  One 8-byte load says that an id is absent, or where it is
// to be found but for ids that share a bit: the entry there is compared, and
// when that is smaller a galloping search goes on from it, so that a clustered
// row only costs a few more steps.  The index (4 bytes per edge + 40 per
// vertex) and the weight summaries (csaw_graph.cu) are built in the call.
//
// Measured (RMAT s20 ef32, 1 M walkers, 40 steps): 150 ms with the index's
// construction (2.6 ms) against 459 ms for the streaming kernel.  Bound by
// instruction issue and dependent loads together (24 or 40 warps per SM instead
// of 32 are 7-9 % slower).
#include <atomic>
#include <cmath>

#include "csaw_internal.cuh"

namespace csaw {

constexpr int N2V_THREADS = 256;
constexpr int N2V_WARPS = N2V_THREADS / 32;
constexpr uint32_t N2V_SLOTS = 32;            // slots a warp keeps sums of
constexpr int N2V_U = 4;                      // list ids per lane and round
constexpr int N2V_B = 2;                      // look-ups per lane and batch
constexpr uint32_t N2V_BATCH = 32 * N2V_B;
constexpr uint32_t N2V_PREV = 0xFFFFFFFFu, N2V_NONE = 0xFFFFFFFEu;   // queue marks: prev itself, no entry
constexpr uint32_t N2V_QUEUE = 32 * N2V_U + N2V_BATCH;
constexpr uint32_t N2V_HOLD = 4;               // batches whose common neighbours are held
constexpr uint32_t N2V_HELD = N2V_HOLD * N2V_BATCH;

// Row v's index: the ids' span [first, first + span] in at most 2^k ranges of
// 2^shift ids, k = floor(log2(d)) + N2V_SPREAD, in words {ids before the word,
// bits} from word (off[v] >> N2V_PACK) + v; the next row's start at least
// floor(d >> N2V_PACK) + 1 >= max(1, 2^k / 32) words later.  The count of a
// word without bits is never read.  rec[v] = {row start, row end, weight sum,
// first | span << 32}.
constexpr uint32_t N2V_SPREAD = 4;
constexpr uint32_t N2V_PACK = 5 - N2V_SPREAD;

__device__ __forceinline__ uint32_t n2v_shift(uint32_t d, uint32_t span)
{
    const uint32_t k = 31u + N2V_SPREAD - (uint32_t)__clz(d);   // d > 0
    const uint32_t bits = 32u - (uint32_t)__clz(span);
    return bits > k ? bits - k : 0u;
}

__device__ __forceinline__ uint64_t n2v_index_at(uint64_t beg, uint32_t v) { return (beg >> N2V_PACK) + v; }

static uint64_t n2v_index_words(uint64_t E, uint64_t V) { return (E >> N2V_PACK) + V + 1; }

constexpr uint32_t N2V_BIG_ROW = 4096;   // rows above this are filled by a whole block

// Thread t of nt fills the (zeroed) index words of one row.
__device__ __forceinline__ void n2v_fill_row(const uint32_t* __restrict__ row, uint32_t d, uint2* __restrict__ index,
                                             uint32_t t, uint32_t nt)
{
    const uint32_t first = __ldg(row), shift = n2v_shift(d, __ldg(row + d - 1) - first);
    for (uint32_t i = t; i < d; i += nt) {
        const uint32_t b = (__ldg(row + i) - first) >> shift;
        uint2* word = index + (b >> 5);
        atomicOr(&word->y, 1u << (b & 31));
        if (i == 0 || ((__ldg(row + i - 1) - first) >> shift) >> 5 != b >> 5) word->x = i;
    }
}

// sums: the weights' per-vertex records, or null (all weights one).
__global__ void __launch_bounds__(256) n2v_index_kernel(const uint64_t* __restrict__ off,
                                                        const uint32_t* __restrict__ col,
                                                        const uint64_t* __restrict__ sums, uint32_t V,
                                                        uint2* __restrict__ index, uint64_t* __restrict__ rec,
                                                        uint32_t* __restrict__ big, unsigned long long* __restrict__ n_big)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t gw = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t v = gw; v < V; v += nw) {
        const uint64_t beg = __ldg(off + v), end = __ldg(off + v + 1);
        const uint32_t d = (uint32_t)(end - beg);
        if (lane == 0) {
            ulonglong2* r = reinterpret_cast<ulonglong2*>(rec + 4 * v);
            uint64_t ids = 0;
            if (d) {
                const uint32_t first = __ldg(col + beg);
                ids = first | (uint64_t)(__ldg(col + end - 1) - first) << 32;
            }
            r[0] = make_ulonglong2(beg, end);
            r[1] = make_ulonglong2(sums ? __ldg(sums + 4 * v + 2) : (uint64_t)d, ids);
            if (d > N2V_BIG_ROW) big[atomicAdd(n_big, 1ull)] = (uint32_t)v;
        }
        if (d && d <= N2V_BIG_ROW) n2v_fill_row(col + beg, d, index + n2v_index_at(beg, (uint32_t)v), lane, 32u);
    }
}

__global__ void __launch_bounds__(1024) n2v_index_big_kernel(const uint64_t* __restrict__ off,
                                                             const uint32_t* __restrict__ col,
                                                             uint2* __restrict__ index, const uint32_t* __restrict__ big,
                                                             const unsigned long long* __restrict__ n_big)
{
    const unsigned long long n = *n_big;
    for (unsigned long long k = blockIdx.x; k < n; k += gridDim.x) {
        const uint32_t v = big[k];
        const uint64_t beg = __ldg(off + v);
        n2v_fill_row(col + beg, (uint32_t)(__ldg(off + v + 1) - beg), index + n2v_index_at(beg, v), threadIdx.x,
                     blockDim.x);
    }
}

struct N2vParams {
    const uint32_t* __restrict__ col;
    const uint32_t* __restrict__ w;      // null: all weights one
    uint64_t E;
    CdfView c;                           // summaries of the weights (null without weights)
    const uint2* __restrict__ index;
    const uint64_t* __restrict__ rec;
    uint32_t V;
    const uint32_t* __restrict__ starts;
    uint64_t n;
    uint32_t L;
    uint32_t* __restrict__ path;
    PhiloxKeys keys;
    uint32_t m0, m1, m2;
    uint32_t tele, tele_q32;
    unsigned long long* next_walker;
};

// A neighbour list and its index.
struct N2vRow {
    const uint32_t* a;      // ids
    const uint2* index;
    uint64_t beg;
    uint32_t d;
    uint32_t first, span;   // of the ids
    uint32_t shift;
};

__device__ __forceinline__ N2vRow n2v_row(const N2vParams& p, uint32_t v, ulonglong2 ends, uint64_t ids)
{
    N2vRow r;
    r.beg = ends.x;
    r.d = (uint32_t)(ends.y - ends.x);
    r.a = p.col + r.beg;
    r.index = p.index + n2v_index_at(r.beg, v);
    r.first = (uint32_t)ids;
    r.span = (uint32_t)(ids >> 32);
    r.shift = n2v_shift(r.d, r.span);
    return r;
}

// The range of id u (an id outside the row's span: the last one).
__device__ __forceinline__ uint32_t n2v_range(const N2vRow& r, uint32_t u)
{
    return min(u - r.first, r.span) >> r.shift;
}

// Whether row r may hold id u of range b, and the first position it can be at.
__device__ __forceinline__ bool n2v_guess(const N2vRow& r, uint32_t u, uint32_t b, uint2 word, uint32_t* at)
{
    const uint32_t bit = 1u << (b & 31);
    *at = word.x + __popc(word.y & (bit - 1u));
    return (word.y & bit) != 0u && u - r.first <= r.span;
}

// The row's weight prefix sum up to position i (inclusive).
__device__ __forceinline__ uint64_t n2v_W(const N2vParams& p, uint64_t beg, uint32_t i)
{
    if (!p.w) return (uint64_t)i + 1;
    const uint64_t e = beg + i, gb = e & ~7ull;
    uint64_t s = gb > beg ? __ldg(p.c.s1 + (gb >> 3) - 1) : 0ull;
    const uint4 x = __ldg(reinterpret_cast<const uint4*>(p.w + gb));
    const uint4 y = __ldg(reinterpret_cast<const uint4*>(p.w + gb) + 1);
    const uint32_t v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (gb + j >= beg && gb + j <= e) s += v[j];
    return s;
}

template <bool WIDE>
struct N2vAcc { using T = uint32_t; };
template <>
struct N2vAcc<true> { using T = uint64_t; };

template <bool WIDE>
__device__ __forceinline__ uint64_t n2v_sum(uint32_t x)
{
    if constexpr (WIDE) return warp_sum_u64(x);
    else return (uint64_t)__reduce_add_sync(CSAW_FULL_MASK, x);
}

// A warp's shared buffers.
template <bool WIDE>
struct N2vShared {
    uint64_t cum[N2V_SLOTS];      // weight sum of the common neighbours up to the slot's end
    typename N2vAcc<WIDE>::T jw[N2V_HELD];   // common neighbours held: running weight sum and position in N(cur)
    // ids whose bit is set, their index in the list (N2V_PREV: prev itself)
    // and the first position to compare
    uint2 at[N2V_QUEUE];
    uint32_t id[N2V_QUEUE];
    uint32_t pos[N2V_SLOTS];      // 1 + position in N(cur) of the slot's last common neighbour
    uint32_t from[N2V_SLOTS];     // list index of the slot's first queue entry
    uint32_t jpos[N2V_HELD];
};

// One step: the position in N(cur) of the pick for draw r; false at a dead
// end.  cur/prev: the two lists; total: the row's weight sum.
// WIDE: the sum of N2V_HELD weights may pass 2^32.
//
// The shorter list is read 32 * N2V_U ids at a time; ids whose bit is
// set in the longer list's index queue up, and N2V_BATCH queued ids at a time are
// looked up exactly.  The common neighbours of the first N2V_HOLD batches are held, and
// the pick is searched with them.  A step with more batches keeps, per slot
// of G batches, the running weight sum and the last common position, which is
// enough to place the draw in one slot; that slot's batches are then formed
// again.  A step is a chain of dependent loads (list, index; entries, weights), so what counts is how few links it has: several ids per lane and
// round, and several compared per lane and batch, go through each link
// together.
template <bool WIDE>
__device__ __forceinline__ bool n2v_pick(const N2vParams& p, const N2vRow& cur, const N2vRow& prev, uint32_t prev_id,
                                         uint64_t total, uint64_t r, N2vShared<WIDE>& sh, int lane, uint32_t* idx)
{
    const bool own = cur.d <= prev.d;
    const uint32_t* list = own ? cur.a : prev.a;
    const uint32_t n = own ? cur.d : prev.d;
    const N2vRow other = own ? prev : cur;
    const uint32_t* lw = p.w ? p.w + cur.beg : nullptr;
    const uint32_t lt = lanemask_lt();
    const uint32_t G = (n / N2V_BATCH + N2V_SLOTS) / N2V_SLOTS;   // batches per slot: at most n / N2V_BATCH + 1 batches
    const uint64_t m2 = p.m2;
    const uint64_t dm1 = (uint64_t)p.m1 - m2;   // wrapping differences
    uint64_t run = 0, dp = 0, x = 0, before = 0;
    typename N2vAcc<WIDE>::T held = 0;   // weight sum of those held
    uint32_t pp = 0xFFFFFFFFu, last_pos = 0, batch = 0, n_batches = 0, j0 = 0, from = 0, to = cur.d, nj = 0;
    auto S_at = [&](uint32_t pe, uint64_t cum) -> uint64_t {   // S of the first pe positions
        return pe == 0 ? 0ull : m2 * n2v_W(p, cur.beg, pe - 1) + dm1 * cum + (pp < pe ? dp : 0ull);
    };
#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
        // queued entries are queue[head .. qn); the current slot and the
        // batches that it still takes
        uint32_t head = 0, qn = 0, slot = 0, left = G;
        if (!own && j0 == 0) {
            // where prev itself stands in N(cur)
            const uint32_t b = n2v_range(cur, prev_id);
            uint32_t at;
            if (n2v_guess(cur, prev_id, b, __ldg(cur.index + (b >> 5)), &at)) {
                if (lane == 0) {
                    sh.at[0] = make_uint2(N2V_PREV, at);
                    sh.id[0] = prev_id;
                }
                qn = 1;
            }
        }
        bool placed = false;
        while (!placed) {
            uint32_t u[N2V_U];
            uint2 word[N2V_U];
#pragma unroll
            for (int t = 0; t < N2V_U; ++t) {
                const uint32_t j = j0 + 32u * t + lane;
                u[t] = j < n ? __ldg(list + j) : 0u;
            }
#pragma unroll
            for (int t = 0; t < N2V_U; ++t)
                word[t] = __ldg(other.index + (n2v_range(other, u[t]) >> 5));
#pragma unroll
            for (int t = 0; t < N2V_U; ++t) {
                if (j0 + 32u * t < n) {
                    const uint32_t j = j0 + 32u * t + lane;
                    uint32_t at;
                    bool may = n2v_guess(other, u[t], n2v_range(other, u[t]), word[t], &at);
                    if (u[t] == prev_id) may = own;
                    may = may && j < n;
                    const uint32_t b = __ballot_sync(CSAW_FULL_MASK, may);
                    if (may) {
                        const uint32_t k = qn + __popc(b & lt);
                        sh.at[k] = make_uint2(j, at);
                        sh.id[k] = u[t];
                    }
                    qn += __popc(b);
                }
            }
            j0 += 32u * N2V_U;
            __syncwarp();
            const bool last = j0 >= n;
            while (head + N2V_BATCH <= qn || (last && head < qn)) {
                uint32_t j[N2V_B], pos[N2V_B], jb[N2V_B], val[N2V_B], id[N2V_B], there[N2V_B];
                if (left == G && lane == 0) sh.from[slot] = sh.at[head].x;
                // compared entry and weight are loaded together, for all of
                // the lane's ids
#pragma unroll
                for (int t = 0; t < N2V_B; ++t) {
                    const uint32_t k = head + 32u * t + lane;
                    const bool ok = k < qn;
                    const uint2 q = ok ? sh.at[k] : make_uint2(N2V_NONE, 0u);
                    id[t] = ok ? sh.id[k] : 0u;
                    j[t] = q.x;
                    pos[t] = q.y;
                    there[t] = __ldg(other.a + pos[t]);
                    val[t] = lw ? __ldg(lw + (own && ok ? j[t] : pos[t])) : 1u;
                }
                // where ids share a bit: on to the first entry that is not smaller
                bool more = true;
                for (int step = 0; more && step < 4; ++step) {
                    more = false;
#pragma unroll
                    for (int t = 0; t < N2V_B; ++t) {
                        if (there[t] < id[t] && pos[t] < other.d) {
                            ++pos[t];
                            there[t] = pos[t] < other.d ? __ldg(other.a + pos[t]) : 0xFFFFFFFFu;
                            if (!own && lw) val[t] = __ldg(lw + pos[t]);
                        }
                        more |= there[t] < id[t] && pos[t] < other.d;
                    }
                }
                if (more) {
#pragma unroll 1
                    for (int t = 0; t < N2V_B; ++t) {
                        uint32_t u1 = id[0], c = there[0], lo = pos[0];
#pragma unroll
                        for (int t2 = 1; t2 < N2V_B; ++t2)
                            if (t == t2) { u1 = id[t2]; c = there[t2]; lo = pos[t2]; }
                        if (c >= u1 || lo >= other.d) continue;
                        uint32_t hi = lo + 1;
                        for (uint32_t step = 1; hi < other.d && __ldg(other.a + hi) < u1; step <<= 1) {
                            lo = hi;
                            hi = min(lo + 2 * step, other.d);
                        }
                        while (lo + 1 < hi) {
                            const uint32_t mid = (lo + hi) >> 1;
                            if (__ldg(other.a + mid) < u1) lo = mid; else hi = mid;
                        }
                        c = hi < other.d ? __ldg(other.a + hi) : 0xFFFFFFFFu;
#pragma unroll
                        for (int t2 = 0; t2 < N2V_B; ++t2)
                            if (t == t2) {
                                pos[t2] = hi;
                                there[t2] = c;
                                if (!own && lw) val[t2] = __ldg(lw + hi);
                            }
                    }
                }
#pragma unroll
                for (int t = 0; t < N2V_B; ++t) {
                    const bool ok = j[t] != N2V_NONE;
                    const bool hit = ok && there[t] == id[t] && pos[t] < other.d;
                    const bool is_prev = ok && id[t] == prev_id;
                    if (own) pos[t] = j[t];
                    const uint32_t bp = __ballot_sync(CSAW_FULL_MASK, is_prev && (own || hit));
                    if (bp) {
                        const int l = __ffs(bp) - 1;
                        pp = __shfl_sync(CSAW_FULL_MASK, pos[t], l);
                        dp = ((uint64_t)p.m0 - m2) * __shfl_sync(CSAW_FULL_MASK, val[t], l);
                    }
                    jb[t] = __ballot_sync(CSAW_FULL_MASK, hit && !is_prev);
                    if (!hit || is_prev) val[t] = 0u;
                }
                head += N2V_BATCH;
                ++batch;
                --left;
                uint64_t after = run;
                uint32_t end_pos = last_pos;   // positions ascend over the common neighbours
#pragma unroll
                for (int t = 0; t < N2V_B; ++t) {
                    if (jb[t]) {
                        after += n2v_sum<WIDE>(val[t]);
                        end_pos = __shfl_sync(CSAW_FULL_MASK, pos[t], 31 - __clz(jb[t])) + 1u;
                    }
                }
                if (phase == 1) {
                    // a slot's batches in turn, until the one that holds x
                    const uint32_t pe = batch == n_batches ? cur.d : end_pos;
                    placed = batch == n_batches || left == 0 || S_at(pe, after) > x;
                    if (placed) {
                        before = run;
                        from = last_pos;
                        to = pe;
                    }
                } else {
                    if (lane == 0) {
                        sh.cum[slot] = after;
                        sh.pos[slot] = end_pos;
                    }
                    if (left == 0) {
                        ++slot;
                        left = G;
                    }
                }
                if (phase == 0 ? batch <= N2V_HOLD : placed) {
                    if (phase == 1) {
                        nj = 0;
                        held = 0;
                    }
#pragma unroll
                    for (int t = 0; t < N2V_B; ++t) {
                        if (jb[t] == 0) continue;
                        typename N2vAcc<WIDE>::T incl = val[t];
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const auto y = __shfl_up_sync(CSAW_FULL_MASK, incl, o);
                            if (lane >= o) incl += y;
                        }
                        if ((jb[t] >> lane) & 1u) {
                            const uint32_t k = nj + __popc(jb[t] & lt);
                            sh.jpos[k] = pos[t];
                            sh.jw[k] = held + incl;
                        }
                        held += __shfl_sync(CSAW_FULL_MASK, incl, 31);
                        nj += __popc(jb[t]);
                    }
                }
                if (placed) break;
                run = after;
                last_pos = end_pos;
            }
            if (last) break;
            // the rest of the queue to its front
            if (head) {
                uint2 rest[N2V_B];
                uint32_t rest_id[N2V_B];
#pragma unroll
                for (int t = 0; t < N2V_B; ++t) {
                    const uint32_t k = min(head + 32u * t + lane, N2V_QUEUE - 1);
                    rest[t] = sh.at[k];
                    rest_id[t] = sh.id[k];
                }
                __syncwarp();
                qn -= head;
                head = 0;
#pragma unroll
                for (int t = 0; t < N2V_B; ++t) {
                    if (32u * t + lane < qn && !placed) {
                        sh.at[32u * t + lane] = rest[t];
                        sh.id[32u * t + lane] = rest_id[t];
                    }
                }
            }
        }
        __syncwarp();
        if (phase == 1) break;
        n_batches = batch;
        const uint64_t T = m2 * total + dm1 * run + dp;
        if (T == 0) return false;
        x = scale_draw(r, T);
        if (batch <= N2V_HOLD) break;
        // the slot: the first whose end exceeds x (the last slot's end is T)
        const uint32_t n_slots = slot + (left < G ? 1u : 0u);
        if (lane == 0) sh.pos[n_slots - 1] = cur.d;
        __syncwarp();
        const uint32_t per = (n_slots + 31) >> 5;
        const uint32_t mine = min(per * (lane + 1), n_slots) - 1;
        const uint32_t b1 = __ballot_sync(CSAW_FULL_MASK, S_at(sh.pos[mine], sh.cum[mine]) > x);
        uint32_t in_slot = per * ((uint32_t)__ffs(b1) - 1);
        if (per > 1) {
            const uint32_t s = min(in_slot + lane, n_slots - 1);
            const uint32_t b2 = __ballot_sync(CSAW_FULL_MASK, S_at(sh.pos[s], sh.cum[s]) > x);
            in_slot = min(in_slot + (uint32_t)__ffs(b2) - 1, n_slots - 1);
        }
        run = in_slot ? sh.cum[in_slot - 1] : 0ull;
        last_pos = in_slot ? sh.pos[in_slot - 1] : 0u;
        j0 = in_slot ? sh.from[in_slot] : 0u;
        batch = in_slot * G;
        __syncwarp();
    }
    // positions [from, to) of N(cur) hold the pick; the common neighbours at
    // them are held, ascending, `before` the weight sum of earlier ones
    auto S = [&](uint32_t i, uint64_t W) -> uint64_t {
        uint32_t lo = 0, hi = nj;   // common neighbours at positions <= i
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (sh.jpos[mid] <= i) lo = mid + 1; else hi = mid;
        }
        return m2 * W + dm1 * (before + (lo ? (uint64_t)sh.jw[lo - 1] : 0ull)) + (pp <= i ? dp : 0ull);
    };
    // the 8-edge group (numbered from the row's first): S at a group's end
    // needs a summary entry alone
    const uint64_t g0 = cur.beg >> 3;
    const uint32_t skew = (uint32_t)(cur.beg & 7u);   // the row's first place in its first group
    uint32_t glo = (skew + from) >> 3, ghi = (uint32_t)(((uint64_t)skew + to - 1) >> 3);
    while (glo < ghi) {
        // first g in [glo, ghi) whose end exceeds x, else ghi; 32 probes at a time
        const uint32_t step = (ghi - glo + 31) >> 5;
        const uint32_t g = glo + step * (lane + 1) - 1;
        const bool in = g < ghi;
        bool above = false;
        if (in) {
            const uint32_t i = 8 * g + 7 - skew;
            above = S(i, p.w ? __ldg(p.c.s1 + g0 + g) : (uint64_t)i + 1) > x;
        }
        const uint32_t probed = __popc(__ballot_sync(CSAW_FULL_MASK, in));
        const uint32_t b = __ballot_sync(CSAW_FULL_MASK, above);
        if (b) {
            const uint32_t k = (uint32_t)__ffs(b) - 1;
            ghi = glo + step * (k + 1) - 1;
            glo += step * k;
        } else {
            glo += step * probed;   // every probe was at or below x
        }
    }
    const uint32_t e = 8 * glo + (lane & 7);   // place of a position plus skew
    const bool in = e >= skew + from && e - skew < to;
    const uint32_t i = in ? e - skew : from;
    const uint32_t hit = __ballot_sync(CSAW_FULL_MASK, lane < 8 && in && S(i, n2v_W(p, cur.beg, i)) > x);
    *idx = hit ? 8 * glo + (uint32_t)(__ffs(hit) - 1) - skew : to - 1;
    __syncwarp();
    return true;
}

template <bool WIDE, bool TELE>
__global__ void __launch_bounds__(N2V_THREADS, 4) walk_n2v_kernel(N2vParams p)
{
    __shared__ N2vShared<WIDE> s_warp[N2V_WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t row_len = (uint64_t)p.L + 1;
    while (true) {
        unsigned long long wk = 0;
        if (lane == 0) wk = atomicAdd(p.next_walker, 1ull);
        wk = __shfl_sync(CSAW_FULL_MASK, wk, 0);
        if (wk >= p.n) break;
        uint32_t* out = p.path + wk * row_len;
        const uint32_t start = __ldg(p.starts + wk);
        if (start >= p.V) {
            for (uint64_t t = lane; t < row_len; t += 32) out[t] = CSAW_NONE;
            continue;
        }
        uint32_t cur = start, prev_id = CSAW_NONE;
        N2vRow prev = {};
        uint32_t buf = lane == 0 ? cur : CSAW_NONE;
        uint64_t flushed = 0;
        for (uint32_t s = 0; s < p.L; ++s) {
            uint32_t nxt = 0;
            bool jump = false;
            if constexpr (TELE)
                jump = (uint32_t)(philox_draw(p.keys, 1u, cur, s, (uint32_t)wk) >> 32) < p.tele_q32;
            if (!jump) {
                const ulonglong2* rc = reinterpret_cast<const ulonglong2*>(p.rec + 4ull * cur);
                const ulonglong2 ends = __ldg(rc), sum_ids = __ldg(rc + 1);
                const uint64_t total = sum_ids.x;
                const N2vRow row = n2v_row(p, cur, ends, sum_ids.y);
                const uint64_t r = philox_draw(p.keys, 0u, cur, s, (uint32_t)wk);
                uint32_t idx = 0;
                bool moved = row.d != 0;
                if (moved && prev_id == CSAW_NONE) {
                    // no previous vertex: the weights alone
                    moved = total != 0;
                    if (moved) {
                        const uint64_t x = scale_draw(r, total);
                        idx = p.w ? (uint32_t)(w_search<true>(p.c, p.w, p.E, ends.x, ends.y, x) - ends.x) : (uint32_t)x;
                    }
                } else if (moved) {
                    moved = n2v_pick<WIDE>(p, row, prev, prev_id, total, r, s_warp[wid], lane, &idx);
                }
                __syncwarp();
                if (moved) {
                    nxt = __ldg(row.a + idx);
                    prev_id = cur;
                    prev = row;
                } else {
                    if constexpr (!TELE) break;
                    jump = true;   // a dead end teleports
                }
            }
            if constexpr (TELE) {
                if (jump) {
                    nxt = p.tele == CSAW_TELEPORT_RESTART
                              ? start
                              : (uint32_t)scale_draw(philox_draw(p.keys, 2u, cur, s, (uint32_t)wk), p.V);
                    prev_id = CSAW_NONE;
                }
            }
            cur = nxt;
            const uint64_t t = (uint64_t)s + 1;
            if ((uint32_t)(t & 31) == (uint32_t)lane) buf = cur;
            if ((t & 31) == 31) {
                out[t - 31 + lane] = buf;
                buf = CSAW_NONE;
                flushed = t + 1;
            }
        }
        for (uint64_t t = flushed + lane; t < row_len; t += 32)
            out[t] = (t < flushed + 32) ? buf : CSAW_NONE;
    }
}

template <bool WIDE, bool TELE>
static csaw_status launch_n2v_k(const N2vParams& p, int sm_count, cudaStream_t s)
{
    static std::atomic<int> cached{0};
    int per_sm = cached.load(std::memory_order_acquire);
    if (per_sm == 0) {
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, walk_n2v_kernel<WIDE, TELE>,
                                                                      N2V_THREADS, 0);
        if (e != cudaSuccess) return cuda_fail(e, "occupancy(walk_n2v)");
        if (per_sm < 1) per_sm = 1;
        cached.store(per_sm, std::memory_order_release);
    }
    uint64_t blocks = (p.n + N2V_WARPS - 1) / N2V_WARPS;
    const uint64_t cap = (uint64_t)sm_count * per_sm;
    if (blocks > cap) blocks = cap;
    walk_n2v_kernel<WIDE, TELE><<<(unsigned)blocks, N2V_THREADS, 0, s>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "walk_n2v_kernel launch");
    return CSAW_OK;
}

uint64_t n2v_bytes(const csaw_graph* g)
{
    const uint64_t sums = g->w && !g->cdf[CSAW_BIAS_EDGE_WEIGHT] ? sizeof(uint64_t) * wsum_layout(g->E, g->V).words : 0;
    return sums + sizeof(uint2) * n2v_index_words(g->E, g->V) + sizeof(uint64_t) * (4 * (uint64_t)g->V + 1) +
           sizeof(uint32_t) * (g->E / N2V_BIG_ROW + 2);
}

// Streaming, a step costs by the row it stands on, one that an edge led to;
// over the index, by the shorter of two rows' lists, which stays near the mean
// degree however long the hubs are.  So the index pays where the rows that
// walks come to are longer than the mean, once its construction is paid, and
// hardly ever on a regular graph, where both lists are alike (degree 4: 0.64 ns
// a step streamed and 0.83 over the index with the chip full; 64: 1.04 and
// 1.13; 512 of which half are common: 2.85 and 4.49).  RMAT s12 1.41 and 0.99,
// s16 2.9 and 1.2, s20 5.8 and 2.4; 16 stars of 60,000 leaves 35 and 1.0.  Each
// side is what its steps cost with the chip full and what the slowest walker
// takes besides, however few walk beside it.
// The figures, in ps, are fitted to the choices, not to either side alone (a
// neighbour held to cost the index 1.4 to 1.6 times as much as streaming, as on
// the regular rows of 512): 1,087 calls on 37 graphs (grids, circulants,
// cliques, random, Zipf, log-normal, preferential attachment, bipartite, stars,
// RMAT s12 to s21), 16 to 1,000,000 walkers of 2 to 120 steps.  Of those 10
// take longer than streamed by more than 4 %, at most by 21.
bool n2v_index_pays(const csaw_graph* g, uint64_t n, uint32_t length)
{
    if (g->E == 0 || g->max_degree > 0x7FFFFFFFu) return false;   // positions plus 8 fit 32 bits
    if (n2v_bytes(g) > array_room()) return false;
    const double walkers = (double)n, steps = (double)length, mean = (double)g->E / (double)g->V;
    const double slowest = slowest_walk(g, walkers, steps, g->reach, 0.638 * g->reach_spread);
    const double streamed = walkers * steps * (15.6 + 4.42 * g->reach) + 0.938e6 * steps + 5.14e3 * slowest;
    const double indexed = 38.9 * (double)g->E + 46.3e6 + walkers * steps * (410.0 + 6.26 * mean) +
                           (0.466e6 + 8.2e3 * mean) * steps;
    return streamed >= indexed;
}

csaw_status walk_n2v(const csaw_graph* g, const csaw_bias* bias, uint64_t max_bias, const uint32_t* starts, uint64_t n,
                     uint32_t length, uint64_t rng_seed, uint32_t tele, uint32_t tele_q32, uint32_t* path,
                     unsigned long long* next_walker, cudaStream_t s, bool* done)
{
    *done = false;
    void *sums = nullptr, *index = nullptr, *rec = nullptr, *big = nullptr;
    N2vParams p;
    const uint64_t* kept = g->w ? g->cdf[CSAW_BIAS_EDGE_WEIGHT] : nullptr;
    const uint64_t n_big = g->E / N2V_BIG_ROW + 2;   // rows above N2V_BIG_ROW, then their count
    csaw_status st = CSAW_OK;
    if (g->w && !kept) st = dalloc(&sums, sizeof(uint64_t) * wsum_layout(g->E, g->V).words, s);
    const size_t index_bytes = sizeof(uint2) * n2v_index_words(g->E, g->V);
    if (st == CSAW_OK) st = dalloc(&index, index_bytes, s);
    if (st == CSAW_OK) st = dalloc(&rec, sizeof(uint64_t) * 4 * (uint64_t)g->V, s);
    if (st == CSAW_OK) st = dalloc(&big, sizeof(uint64_t) + sizeof(uint32_t) * n_big, s);
    if (st == CSAW_OK && g->w) {
        p.c = kept ? cdf_view(kept, g->E, g->V) : wsum_view((const uint64_t*)sums, g->E, g->V);
        if (!kept)
            st = enqueue_cdf_build_raw(g->off, g->col, g->w, g->deg, g->V, g->E, g->sm_count, CSAW_BIAS_EDGE_WEIGHT,
                                       nullptr, (uint64_t*)p.c.s1, (uint64_t*)p.c.s2, (uint64_t*)p.c.rec, s);
    }
    if (st == CSAW_OK) {
        unsigned long long* big_n = (unsigned long long*)big;
        uint32_t* big_rows = (uint32_t*)(big_n + 1);
        cudaError_t e = cudaMemsetAsync(big_n, 0, sizeof(*big_n), s);
        if (e == cudaSuccess) e = cudaMemsetAsync(index, 0, index_bytes, s);
        if (e == cudaSuccess) {
            uint64_t blocks = ((uint64_t)g->V + 7) / 8;
            const uint64_t cap = (uint64_t)g->sm_count * 8;
            if (blocks > cap) blocks = cap;
            n2v_index_kernel<<<(unsigned)blocks, 256, 0, s>>>(g->off, g->col, g->w ? p.c.rec : nullptr, g->V,
                                                             (uint2*)index, (uint64_t*)rec, big_rows, big_n);
            if (g->max_degree > N2V_BIG_ROW)
                n2v_index_big_kernel<<<(unsigned)g->sm_count * 2, 1024, 0, s>>>(g->off, g->col, (uint2*)index, big_rows,
                                                                               big_n);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) st = cuda_fail(e, "n2v_index_kernel launch");
        p.col = g->col; p.w = g->w; p.E = g->E;
        p.index = (const uint2*)index; p.rec = (const uint64_t*)rec;
        p.V = g->V; p.starts = starts; p.n = n; p.L = length; p.path = path;
        p.keys = philox_round_keys(rng_seed);
        p.m0 = bias->n2v_mult[0]; p.m1 = bias->n2v_mult[1]; p.m2 = bias->n2v_mult[2];
        p.tele = tele; p.tele_q32 = tele_q32;
        p.next_walker = next_walker;
        const bool wide = max_bias * N2V_HELD >= (1ull << 32);
        if (st == CSAW_OK)
            st = tele ? (wide ? launch_n2v_k<true, true>(p, g->sm_count, s) : launch_n2v_k<false, true>(p, g->sm_count, s))
                      : (wide ? launch_n2v_k<true, false>(p, g->sm_count, s) : launch_n2v_k<false, false>(p, g->sm_count, s));
    }
    dfree(sums, s);
    dfree(index, s);
    dfree(rec, s);
    dfree(big, s);
    *done = st == CSAW_OK;
    if (st == CSAW_ERR_NOMEM) {
        // no room for the index, the sums or the sums' own temporaries: the
        // caller streams the rows
        clear_error();
        return CSAW_OK;
    }
    return st;
}

}  // namespace csaw
