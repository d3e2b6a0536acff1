// k_walk: the RANGE search for instances of a few thousand timestamps of up to 128 workers, a warp per instance, in one launch.
// Nothing is sorted and no barrier but the warp's own is passed.
//
// The best selection whose minimum is at time t has max(Z) = G(t) = max over the rows of their first element at or after t.
// The timeline up to the first exhausted row is cut into a few hundred cells.  One pass over the elements (a maximum of `next`
// per cell, then a prefix maximum) gives G at every cell's start: every candidate of a cell has d >= G(start) - end, and a
// cell that raises G holds one with d <= G(next start) - start.  A second pass collects the elements that raise G in the
// cells that the smallest of these upper bounds does not discard - a few dozen - and each of them gets its exact d from the
// others of its cell.  More of them than there is room for (many equal times): the rows are walked from barrier to barrier.
#include "zl_batch.cuh"
#include "zl_host.h"

namespace zl {

constexpr int WALK_MAX_R = 256;
constexpr int WALK_MAX_CELLS = 512;
constexpr unsigned WALK_NODES = 128;       // room for candidates

struct WalkParams {
    int n, R, B, stride, cells, words, check_sorted;      // stride: words between rows in shared memory (odd: no bank conflicts by row)
    const int64_t *ts;
    int32_t *idx; int64_t *barrier; int64_t *wait; int32_t *status;
};

// Relative times as 32-bit words in shared memory, or (spans of 2^32 and more) 64-bit values straight from the rows.
struct NarrowRows {
    typedef uint32_t V;
    const uint32_t *x; uint32_t tminlo; int stride;
    static constexpr V INF = 0xffffffffu;
    __device__ __forceinline__ V at(int p, int i) const { return x[p * stride + i] - tminlo; }
    __device__ __forceinline__ static V lowest(V v) { return __reduce_min_sync(FULL, v); }
    __device__ __forceinline__ static V highest(V v) { return __reduce_max_sync(FULL, v); }
};
struct WideRows {
    typedef uint64_t V;
    const int64_t *ts; int64_t tmin; int R;
    static constexpr V INF = ~0ull;
    __device__ __forceinline__ V at(int p, int i) const { return (uint64_t)(ldg64(ts + (size_t)p * R + i) - tmin) + 1; }
    __device__ __forceinline__ static V lowest(V v) { return warp_reduce(v, OpMin()); }
    __device__ __forceinline__ static V highest(V v) { return warp_reduce(v, OpMax()); }
};

// From barrier to barrier: the minimum is the earliest of the rows' current elements, the barrier the latest; the rows that hold
// the minimum move on.  Smallest d and the time of its minimum, the first of equal ones.  K rows a lane.
template <int K, class ROWS>
__device__ __noinline__ void walk(const ROWS rows, int n, int R, typename ROWS::V last, typename ROWS::V &bd, typename ROWS::V &bt) {
    typedef typename ROWS::V V;
    const int lane = threadIdx.x & 31;
    V t[K], hi = 0, d = ROWS::INF, dt = ROWS::INF;
    int i[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        i[k] = 0;
        t[k] = 32 * k + lane < n ? rows.at(32 * k + lane, 0) : ROWS::INF;
        if (32 * k + lane < n) hi = max(hi, t[k]);
    }
    V M = ROWS::highest(hi);
    // every step takes at least one row an element on: fewer than n * R steps
#pragma unroll 1
    while (M != ROWS::INF) {
        V lo = t[0];
#pragma unroll
        for (int k = 1; k < K; ++k) lo = min(lo, t[k]);
        lo = ROWS::lowest(lo);
        if (lo > last) break;
        if (M - lo < d) { d = M - lo; dt = lo; }                  // the same in every lane
        hi = 0;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (t[k] == lo) {
                do { ++i[k]; t[k] = i[k] < R ? rows.at(32 * k + lane, i[k]) : ROWS::INF; } while (t[k] <= lo);
                hi = max(hi, t[k]);
            }
        M = max(M, ROWS::highest(hi));
    }
    bd = d; bt = dt;
}

// Index of row p's first element at or after time t (R: none).
template <class ROWS>
__device__ __forceinline__ int first_from(const ROWS &rows, int p, int R, typename ROWS::V t) {
    int lo = 0, hi = R;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (rows.at(p, mid) < t) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The cells of an instance and what they leave.  cell: `most` (a power of two, at least 64) words plus 32, node: WALK_NODES, both
// the warp's.  False: more candidates than there is room for.
__device__ __forceinline__ bool search_cells(const NarrowRows &rows, int n, int R, uint32_t t0, uint32_t lmin, uint32_t *cell, int most, uint64_t *node,
                                             uint32_t &bd, uint32_t &bt) {
    const int lane = threadIdx.x & 31, N = n * R;
    const int per = most / 32, ps = __ffs(per) - 1;               // a run of cells a lane; cell c sits at c + c / per (no bank conflicts)
    int sh = 0;
    while (((lmin - 1u) >> sh) >= (uint32_t)most) ++sh;
    const int m = (int)((lmin - 1u) >> sh) + 1;                   // cells: cell c holds the times (c << sh) + 1 .. (c + 1) << sh
#pragma unroll 1
    for (int c = lane; c < most + 32; c += 32) cell[c] = t0;
    __syncwarp();
    // cell c becomes the maximum of `next` over its elements
    {
        int r = 0, c = lane;
#pragma unroll 4
        for (int f = lane; f < N; f += 32) {
            while (c >= R) { c -= R; ++r; }
            const uint32_t T = rows.at(r, c);
            const uint32_t nx = c + 1 < R ? rows.at(r, c + 1) : NarrowRows::INF;
            const uint32_t k = (T - 1u) >> sh;
            if (k < (uint32_t)m) {
                uint32_t *w = cell + k + (k >> ps);
                if (*w < nx) atomicMax(w, nx);
            }
            c += 32;
        }
    }
    __syncwarp();
    // ... and then G at its start: the prefix maximum, exclusive; the smallest upper bound on the way
    uint32_t run = 0;
    uint32_t *mine = cell + lane * (per + 1);
#pragma unroll 1
    for (int j = 0; j < per; ++j) run = max(run, mine[j]);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, run, d); if (lane >= d) run = max(run, y); }
    run = __shfl_up_sync(FULL, run, 1);
    run = lane == 0 ? t0 : max(run, t0);
    uint32_t ub = 0xffffffffu;
#pragma unroll 1
    for (int j = 0; j < per; ++j) {
        const int c = lane * per + j;
        const uint32_t v = mine[j], start = ((uint32_t)c << sh) + 1u;
        mine[j] = run;
        // the element that raises G first has d = G(start) - T at most where G(start) is later than it, else 0; all that
        // raise it end at v at the latest
        if (c < m && v > run && v != NarrowRows::INF) ub = min(ub, v - start);
        run = max(run, v);
    }
    ub = __reduce_min_sync(FULL, ub);
    __syncwarp();
    // the elements that raise G in the cells that are left
    unsigned fill = 0;
    {
        int r = 0, c = lane;
#pragma unroll 2
        for (int f0 = 0; f0 < N; f0 += 32) {
            while (c >= R) { c -= R; ++r; }
            bool keep = false;
            uint32_t T = 0, nx = 0;
            if (f0 + lane < N) {
                T = rows.at(r, c);
                nx = c + 1 < R ? rows.at(r, c + 1) : NarrowRows::INF;
                const uint32_t k = (T - 1u) >> sh;
                if (k < (uint32_t)m) {
                    const uint32_t g = cell[k + (k >> ps)], end = min((uint32_t)((uint64_t)(k + 1u) << sh), lmin);
                    keep = nx > g && nx > T && (g <= end || g - end <= ub);
                }
            }
            const unsigned km = __ballot_sync(FULL, keep);
            const unsigned pos = fill + __popc(km & ((1u << lane) - 1u));
            if (keep && pos < WALK_NODES) node[pos] = ((uint64_t)T << 32) | nx;
            fill += __popc(km);
            c += 32;
        }
    }
    if (fill > WALK_NODES) return false;
    __syncwarp();
    uint32_t d = NarrowRows::INF, t = NarrowRows::INF;
#pragma unroll 1
    for (unsigned i = lane; i < fill; i += 32) {
        const uint32_t T = (uint32_t)(node[i] >> 32), k = (T - 1u) >> sh;
        uint32_t g = max(cell[k + (k >> ps)], T);
#pragma unroll 4
        for (unsigned j = 0; j < fill; ++j) {
            const uint32_t tj = (uint32_t)(node[j] >> 32);
            if (tj < T && (tj - 1u) >> sh == k) g = max(g, (uint32_t)node[j]);
        }
        if (g != NarrowRows::INF && (g - T < d || (g - T == d && T < t))) { d = g - T; t = T; }
    }
    bd = __reduce_min_sync(FULL, d);
    bt = __reduce_min_sync(FULL, d == bd ? t : NarrowRows::INF);
    return bd != NarrowRows::INF;                                 // (always, unless rows are not sorted)
}

// Dynamic shared memory: a warp after the other, P.words words each: the rows (n * stride), candidates, cells.
template <int K>
__global__ void __launch_bounds__(128) k_walk(const WalkParams P) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int n = P.n, R = P.R, N = n * R, b = blockIdx.x * nw + warp;
    uint32_t *x = (uint32_t *)smem + (size_t)warp * P.words;
    uint64_t *node = (uint64_t *)(x + ((n * P.stride + 1) & ~1));
    uint32_t *cell = (uint32_t *)(node + WALK_NODES);
    if (b >= P.B) return;
    const int64_t *ts = P.ts + (size_t)b * N;
    // ---- first and last elements: tmin = min_p e^p_1, t0 = max_p e^p_1, lmin = min_p e^p_R, the span
    uint64_t q[4] = {~0ull, 0, ~0ull, 0};                         // order-preserving unsigned images of int64
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int p = 32 * k + lane;
        if (p < n) {
            const uint64_t u = (uint64_t)ldg64(ts + (size_t)p * R) ^ (1ull << 63), w = (uint64_t)ldg64(ts + (size_t)p * R + R - 1) ^ (1ull << 63);
            q[0] = min(q[0], u); q[1] = max(q[1], u); q[2] = min(q[2], w); q[3] = max(q[3], w);
        }
    }
    // ---- the low words of all timestamps into shared memory, on the way the optional check that rows do not decrease
    bool unsorted = false;
    {
        int r = 0, c = lane;                                      // row and column of the lane's element
        bool bad = false;
        int64_t tail = 0;
#pragma unroll 1
        for (int f0 = 0; f0 < N; f0 += 32 * 8) {
            int64_t v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) { const int f = f0 + 32 * u + lane; v[u] = f < N ? ldg64(ts + f) : INT64_MAX; }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int f = f0 + 32 * u + lane;
                while (c >= R) { c -= R; ++r; }
                if (f < N) x[r * P.stride + c] = (uint32_t)(uint64_t)v[u];
                if (P.check_sorted) {
                    int64_t before = (int64_t)shfl_up((uint64_t)v[u], 1);
                    if (lane == 0) before = tail;
                    tail = (int64_t)shfl_idx((uint64_t)v[u], 31);
                    bad |= f < N && c > 0 && v[u] < before;
                }
                c += 32;
            }
        }
        unsorted = P.check_sorted && __any_sync(FULL, bad);
    }
    q[0] = warp_reduce(q[0], OpMin()); q[1] = warp_reduce(q[1], OpMax());
    q[2] = warp_reduce(q[2], OpMin()); q[3] = warp_reduce(q[3], OpMax());
    const int64_t tmin = (int64_t)(q[0] ^ (1ull << 63)), t0 = (int64_t)(q[1] ^ (1ull << 63));
    const int64_t lmin = (int64_t)(q[2] ^ (1ull << 63)), tmax = (int64_t)(q[3] ^ (1ull << 63));
    int status = ZL_OK;
    if (tmin < 0 || tmax >= VALUE_LIMIT || tmax < tmin || lmin < tmin) status = ZL_ERR_INVALID_ARG;   // outside [0, 2^62), or first/last columns out of order
    else if (unsorted) status = ZL_ERR_UNSORTED;
    __syncwarp();
    int64_t bar = INT64_MIN, wt = INT64_MIN;
    int at[K];
#pragma unroll
    for (int k = 0; k < K; ++k) at[k] = -1;
    if (status == ZL_OK) {
        if ((uint64_t)(tmax - tmin) + 1 < 0xfffffffeull) {
            const NarrowRows rows{x, (uint32_t)(uint64_t)tmin - 1u, P.stride};
            const uint32_t last = (uint32_t)(lmin - tmin) + 1u;
            uint32_t d, t;
            if (!search_cells(rows, n, R, (uint32_t)(t0 - tmin) + 1u, last, cell, P.cells, node, d, t)) walk<K>(rows, n, R, last, d, t);
            bar = tmin - 1 + (int64_t)(t + d); wt = (int64_t)d;
#pragma unroll
            for (int k = 0; k < K; ++k) if (32 * k + lane < n) at[k] = first_from(rows, 32 * k + lane, R, t + d + 1u) - 1;
        } else {
            const WideRows rows{ts, tmin, R};
            uint64_t d, t;
            walk<K>(rows, n, R, (uint64_t)(lmin - tmin) + 1, d, t);
            bar = tmin - 1 + (int64_t)(t + d); wt = (int64_t)d;
#pragma unroll
            for (int k = 0; k < K; ++k) if (32 * k + lane < n) at[k] = first_from(rows, 32 * k + lane, R, t + d + 1) - 1;
        }
    }
    if (lane == 0) {
        P.wait[b] = wt;
        P.barrier[b] = bar;
        if (P.status) P.status[b] = status;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) if (32 * k + lane < n) P.idx[(size_t)b * n + 32 * k + lane] = at[k];
}

bool walk_shape(int n, int R) { return n <= 128 && R <= WALK_MAX_R && (long long)n * R <= SMALL_MAX; }

void enqueue_walk(const Pipeline &q, cudaStream_t st) {
    WalkParams P;
    P.n = q.n; P.R = q.R; P.B = q.B; P.stride = q.R | 1; P.check_sorted = (q.flags & ZL_FLAG_CHECK_SORTED) ? 1 : 0;
    P.ts = q.ts; P.idx = q.idx; P.barrier = q.barrier; P.wait = q.wait; P.status = q.status;
    const int warps = q.B > 4 * q.num_sms ? 4 : 1;                // few instances: one on an SM
    // about eight cells an iteration of the slowest worker: fewer leave more candidates, more cost the passes over them
    P.cells = std::max(64, std::min(WALK_MAX_CELLS, pow2_ceil(8 * q.R)));
    P.words = ((q.n * P.stride + 1) & ~1) + 2 * (int)WALK_NODES + P.cells + 32;
    const size_t smem = (size_t)warps * P.words * 4;
    const dim3 grid((q.B + warps - 1) / warps), block(32 * warps);
    const bool early = !((q.pdl_off >> 9) & 1);
    if (q.n <= 32) launch_dep(early, k_walk<1>, grid, block, smem, st, P);
    else if (q.n <= 64) launch_dep(early, k_walk<2>, grid, block, smem, st, P);
    else launch_dep(early, k_walk<4>, grid, block, smem, st, P);
}

cudaError_t walk_limits() {
    cudaError_t e = cudaFuncSetAttribute(k_walk<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_walk<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_walk<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    return e;
}

}  // namespace zl
