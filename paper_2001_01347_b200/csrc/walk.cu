// k_walk: the RANGE search for instances of a few thousand timestamps of up to 128 workers, a warp per instance, in one launch.
// Nothing is sorted and no barrier but the warp's own is passed.
//
// The best selection whose minimum is the element at time T has max(Z) = G(T) = max over the rows of their first element at or
// after T, and only elements whose passing raises G matter.  The timeline up to the first exhausted row is cut into a few
// hundred cells; one pass over the elements (a maximum of `next` per cell, then a prefix maximum) gives G at every cell's
// start and so a lower bound of every element's d.  The element with the smallest bound is evaluated exactly - a row a lane,
// a search in shared memory -, a second pass collects the ones that its d does not discard (a few, rarely dozens), and these
// are evaluated in the order of their bounds until none is left below the smallest d.  More of them than there is room for
// (many equal times): the rows are walked from barrier to barrier.
#include "zl_batch.cuh"
#include "zl_host.h"

namespace zl {

constexpr int WALK_ALONE = 256;            // timestamps of an instance whose passes take a microsecond or two
constexpr int WALK_MAX_CELLS = 512;
constexpr int WALK_PASSES = 24;            // most passes that take a single candidate
constexpr unsigned WALK_NODES = 128;       // room for candidates
constexpr int WALK_PASSES_FINE = 1;        // passes that take single candidates, beyond which the handle's next calls leave the kernel (regular
                                           // instances need none)

struct WalkParams {
    int n, R, B, stride, cells, words, check_sorted;      // stride: words between rows in shared memory: R and one that reads as infinite
    const int64_t *ts;
    int32_t *idx; int64_t *barrier; int64_t *wait; int32_t *status;
    uint32_t *slow, epoch;                                // pinned host memory, or nullptr: set to the call's number by an instance that this
                                                          // kernel is not made for (many equal or nearly equal waits, spans of 2^32 and more)
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
template <int K>
__device__ __forceinline__ bool search_cells(const NarrowRows &rows, int n, int R, uint32_t t0, uint32_t lmin, uint32_t *cell, int most, uint64_t *node,
                                             uint32_t &bd, uint32_t &bt, int &passes) {
    const int lane = threadIdx.x & 31, N = n * rows.stride;       // all words of the rows, one after the other
    const int per = most / 32, ps = __ffs(per) - 1;               // a run of cells a lane; cell c sits at c + c / per (no bank conflicts)
    // T - 1 < lmin, so its cell ((T - 1) * scale) >> 32 is below `most`.  (T = 0, a time before the first elements, is only met in
    // rows that are not sorted; such an element belongs to no cell.)
    const uint32_t scale = (uint32_t)min((uint64_t)0xffffffffu, ((uint64_t)most << 32) / lmin);
    auto cell_at = [&](uint32_t T) { const uint32_t k = __umulhi(T - 1u, scale); return cell + k + (k >> ps); };
#pragma unroll 1
    for (int c = lane; c < most + 32; c += 32) cell[c] = t0;
    __syncwarp();
    // cell c becomes the maximum of `next` over its elements
    {
#pragma unroll 4
        for (int f = lane; f < N; f += 32) {
            const uint32_t T = rows.at(0, f), nx = rows.at(0, f + 1);
            if (T - 1u < lmin) {
                uint32_t *w = cell_at(T);
                if (*w < nx) atomicMax(w, nx);
            }
        }
    }
    __syncwarp();
    // ... and then a lower bound of G inside it: the exclusive prefix maximum; the most promising cell is the one where that
    // exceeds the cell's end by least
    uint32_t best = NarrowRows::INF, start = 0;
    {
        uint32_t run = 0;
        uint32_t *mine = cell + lane * (per + 1);
#pragma unroll 4
        for (int j = 0; j < per; ++j) run = max(run, mine[j]);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, run, d); if (lane >= d) run = max(run, y); }
        run = __shfl_up_sync(FULL, run, 1);
        run = lane == 0 ? t0 : max(run, t0);
#pragma unroll 4
        for (int j = 0; j < per; ++j) {
            const uint32_t v = mine[j], c = (uint32_t)(lane * per + j);
            const uint32_t end = (uint32_t)(((uint64_t)lmin * (c + 1u)) >> (ps + 5)) + 1u;
            const uint32_t l = run > end ? run - end : 0u;
            if (l < best) { best = l; start = (uint32_t)(((uint64_t)lmin * c) >> (ps + 5)) + 1u; }
            mine[j] = run;
            run = max(run, v);
        }
    }
    __syncwarp();
    // a d that is attained: the rows' first elements at or after that cell's start (about: any time up to lmin will do).  With no
    // more than a few hundred elements the passes below have few candidates as it is.
    uint32_t d = NarrowRows::INF, t = NarrowRows::INF;
    if (n * R > WALK_ALONE) {
        const uint32_t l = __reduce_min_sync(FULL, best);
        const int owner = __ffs(__ballot_sync(FULL, best == l)) - 1;
        start = min(__shfl_sync(FULL, start, owner), lmin);
        uint32_t g = 0, m = NarrowRows::INF;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int p = 32 * k + lane;
            if (p < n) {
                const int i = first_from(rows, p, R, start);
                const uint32_t T = i < R ? rows.at(p, i) : NarrowRows::INF;
                g = max(g, T); m = min(m, T);
            }
        }
        g = __reduce_max_sync(FULL, g); m = __reduce_min_sync(FULL, m);
        if (g != NarrowRows::INF) { d = g - m; t = m; }
    }
    // d of the element at time T: all rows' first elements at or after it
    auto exact = [&](uint32_t T) {
        uint32_t g = T;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int p = 32 * k + lane;
            if (p < n) { const int i = first_from(rows, p, R, T); g = max(g, i < R ? rows.at(p, i) : NarrowRows::INF); }
        }
        return __reduce_max_sync(FULL, g);
    };
    // Best first: (bound, time) of the elements, in that order.  A pass over the elements collects those behind the last one
    // evaluated whose bound is below d (or d itself, at an earlier time); while there are more than there is room for, only the first of them is taken.
    uint64_t after = 0;
    unsigned fill = 0;
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        uint64_t first = ~0ull;
        fill = 0;
#pragma unroll 4
        for (int f0 = 0; f0 < N; f0 += 32) {
            bool keep = false;
            uint64_t q = ~0ull;
            if (f0 + lane < N) {
                const uint32_t T = rows.at(0, f0 + lane), nx = rows.at(0, f0 + lane + 1);
                if (T - 1u < lmin) {
                    const uint32_t g = max(*cell_at(T), T), l = g - T;
                    q = ((uint64_t)l << 32) | T;
                    keep = nx > g && (l < d || (l == d && T < t)) && q >= after;
                }
            }
            if (keep) first = min(first, q);
            const unsigned km = __ballot_sync(FULL, keep);
            if (km) {
                const unsigned pos = fill + __popc(km & ((1u << lane) - 1u));
                if (keep && pos < WALK_NODES) node[pos] = q;
                fill += __popc(km);
            }
        }
        __syncwarp();
        passes = pass;
        if (fill <= WALK_NODES) break;
        if (pass >= WALK_PASSES) return false;
        // the lanes' first candidates, best first
        uint64_t lowest = ~0ull;
#pragma unroll 1
        for (int k = 0; k < 32; ++k) {
            const uint32_t l = __reduce_min_sync(FULL, (uint32_t)(first >> 32));
            const uint32_t T = __reduce_min_sync(FULL, (uint32_t)(first >> 32) == l ? (uint32_t)first : NarrowRows::INF);
            if (l > d || l == NarrowRows::INF) break;
            const uint64_t q = ((uint64_t)l << 32) | T;
            lowest = min(lowest, q);
            if (first == q) first = ~0ull;
            const uint32_t g = exact(T);
            if (g != NarrowRows::INF && (g - T < d || (g - T == d && T < t))) { d = g - T; t = T; }
        }
        after = lowest + 1;
    }
#pragma unroll 1
    for (unsigned done = 0; done < fill; ++done) {
        uint64_t q = ~0ull;
        for (unsigned i = lane; i < fill; i += 32) if (node[i] >= after) q = min(q, node[i]);
        const uint32_t l = __reduce_min_sync(FULL, (uint32_t)(q >> 32));
        const uint32_t T = __reduce_min_sync(FULL, (uint32_t)(q >> 32) == l ? (uint32_t)q : NarrowRows::INF);
        if (l > d || l == NarrowRows::INF) break;
        after = (((uint64_t)l << 32) | T) + 1;
        const uint32_t g = exact(T);
        if (g != NarrowRows::INF && (g - T < d || (g - T == d && T < t))) { d = g - T; t = T; }
    }
    bd = d; bt = t;
    return d != NarrowRows::INF;                                  // (always, unless rows are not sorted)
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
#pragma unroll 1
    for (int p = lane; p < n; p += 32) x[p * P.stride + R] = (uint32_t)(uint64_t)tmin - 2u;      // relative: infinite
    __syncwarp();
    int64_t bar = INT64_MIN, wt = INT64_MIN;
    int at[K], passes = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) at[k] = -1;
    if (status == ZL_OK) {
        if ((uint64_t)(tmax - tmin) + 1 < 0xfffffffeull) {
            const NarrowRows rows{x, (uint32_t)(uint64_t)tmin - 1u, P.stride};
            const uint32_t last = (uint32_t)(lmin - tmin) + 1u;
            uint32_t d, t;
            if (!search_cells<K>(rows, n, R, (uint32_t)(t0 - tmin) + 1u, last, cell, P.cells, node, d, t, passes)) walk<K>(rows, n, R, last, d, t);
            bar = tmin - 1 + (int64_t)(t + d); wt = (int64_t)d;
#pragma unroll
            for (int k = 0; k < K; ++k) if (32 * k + lane < n) at[k] = first_from(rows, 32 * k + lane, R, t + d + 1u) - 1;
        } else {
            const WideRows rows{ts, tmin, R};
            uint64_t d, t;
            passes = WALK_PASSES;
            walk<K>(rows, n, R, (uint64_t)(lmin - tmin) + 1, d, t);
            bar = tmin - 1 + (int64_t)(t + d); wt = (int64_t)d;
#pragma unroll
            for (int k = 0; k < K; ++k) if (32 * k + lane < n) at[k] = first_from(rows, 32 * k + lane, R, t + d + 1) - 1;
        }
    }
    if (lane == 0) {
        if (passes > WALK_PASSES_FINE && P.slow) *(volatile uint32_t *)P.slow = P.epoch;
        P.wait[b] = wt;
        P.barrier[b] = bar;
        if (P.status) P.status[b] = status;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) if (32 * k + lane < n) P.idx[(size_t)b * n + 32 * k + lane] = at[k];
}

// A warp's passes over the elements and its few evaluations are one chain: the more elements, the more other warps it needs
// beside it to be worth more than a CTA that sorts the instance, and the rows must be short and not too few for the bounds to
// be tight.  (Instances with many equal or nearly equal waits cost it 5 to 20 times what a CTA that sorts them takes, n=16, R=64 B=1 335-650 us,
// B=1500 340-710, against 30-50: a handle leaves the kernel after such a call, and without a handle only instances of
// at most WALK_ALONE timestamps are given to it.)  Measured in us, this kernel / a CTA an instance: n=16, R=16, B=1 6.2 / 11; n=4, R=80 10 / 17 (B=1), 22 / 50 (4800);
// n=16, R=30 13 / 23 (100), 13 / 21 (600), 22 / 58 (4800); n=32, R=32 14 / 24 (1), 19 / 23 (600), 38 / 84 (4800); n=100, R=10 18 / 15
// (1), 25 / 17 (100), 27 / 34 (600); n=16, R=100 32 / 29 (600), 37 / 40 (1200), 62 / 116 (4800); n=60, R=50 44 / 42 (600), 45 / 68
// (1200); n=128, R=20 57 / 77 (1200); but n=64, R=64 93 / 75 (1200), n=16, R=128 45 / 43 (1200), n=4, R=200 53 / 30 (1200), n=97, R=4 19 / 15 (6), n=2,
// R=28 11 / 7 (522).
bool walk_shape_alone(int n, int R) { return (long long)n * R <= WALK_ALONE && walk_shape(n, R, 1, 1); }

bool walk_shape(int n, int R, int batch, int num_sms) {
    const long long N = (long long)n * R;
    if (n > 128 || R > 100 || (n < 4 && N > 32)) return false;
    return N <= WALK_ALONE || (N <= 2 * WALK_ALONE && (n <= 64 || batch > 4 * num_sms)) || (N <= 4 * WALK_ALONE && R <= 64 && (n <= 32 || batch > 4 * num_sms)) ||
           (N <= (R <= 64 ? 12 : 8) * WALK_ALONE && n >= 8 && batch > 8 * num_sms);
}

void enqueue_walk(const Pipeline &q, cudaStream_t st) {
    WalkParams P;
    P.n = q.n; P.R = q.R; P.B = q.B; P.stride = q.R + 1; P.check_sorted = (q.flags & ZL_FLAG_CHECK_SORTED) ? 1 : 0;
    P.slow = q.fb.hint && q.epoch ? q.fb.hint + 2 : nullptr; P.epoch = q.epoch;
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
