// The cell route, both objectives, stored and predicted rows: no timestamp is sorted until it is known to matter, and of
// most rows only a few are read at all.
//
// The part of an instance's timeline that can hold the answer is cut into cells of a power of two of time units.  The
// search is branch and bound over the cells:
//   RANGE  The best Z whose minimum is at time t has max(Z) = G(t) = max over the rows of their first element at or after t,
//          so d = G(T) - T, and every candidate of a cell has d >= G(start) - end.  G is set by the rows with long
//          iterations: the slowest fifth to half of the rows ("guards": an eighth of the timestamps or so) give a lower bound of G
//          at every cell's start - a maximum per cell, then a prefix maximum.  The cells with the smallest bounds are
//          evaluated exactly (every row is asked for its elements in them: a search from the row's ends, a few loads); the
//          smallest d discards nearly all other cells, and the ones it does not are evaluated the same way, most promising
//          first.  Where the guards leave too many, the other rows are looked through for gaps longer than d: only those can
//          discard a further cell.
//   SUM    wait(T) = n T - S(T), S = sum of the workers' latest elements.  A sum of deltas per cell and a prefix sum give S
//          at every cell's start, so every candidate of a cell has wait >= n start - S(end) and the cell's last element
//          attains at most n end - S(end).  Cells whose lower bound exceeds a wait that is attained are discarded; the few
//          elements of the others are evaluated exactly.  A worker whose last element lies x before the barrier waits x:
//          times at which these waits alone exceed a wait known to be attained are not looked at, so most of a long row of
//          a fast worker is never read.
//
// k_cells does the whole search of an instance in one launch: a cluster of CTAs, each with a slice of the timeline (all
// rows that count there), a share of the rows when rows are asked, and no global scratch.  k_cell_rest runs behind it: the
// segment sweep for the instances it left over (spans of 2^32 or more, more surviving cells or elements than there is room
// for) and the outputs of instances in error; it returns at once when there are none.
//
// Every CTA of a cluster passes the same cluster barriers: whatever a loop or a branch around one depends on is the same
// value in the whole cluster (never the CTA's own number of rows or cells).
#include <cmath>
#include <cooperative_groups.h>

#include "zl_sweep.cuh"
#include "zl_host.h"

namespace cg = cooperative_groups;

namespace zl {

constexpr uint32_t INF32 = 0xffffffffu;
constexpr int CELL_ALIVE = 128;           // most cells of an instance that the bounds may leave
constexpr int CELL_BATCH = 16;            // most cells that the rows are asked for at once
constexpr int CELL_NODES = 1024;          // most elements in those
constexpr int CELL_CLUSTER = 16;          // most CTAs of a cluster
constexpr long long CELL_ASK = 4;         // asking a row for a cell costs about as much as looking through this many of its elements, all cells of a
                                          // batch at once (n=1024, R=1024, B=64, mean of ten seeds 69 us with 16 and half the batch, 63 with 4)
constexpr int CELL_ROUNDS = 4;            // rounds after the first in which more cells may be left than there is room for (regular rows need one or two, SUM
                                          // up to four; with 48, rows of equal periods, n=64, R=128, took 0.5 ms before they were given up)
constexpr int CELL_HOPELESS = 2 * CELL_ALIVE;    // ... and so many are never worth a further round
// Cells evaluated, and eight for every round, beyond which the handle's next calls leave the route: regular rows, over 300 random shapes, need up
// to 33 (RANGE) and 87 (SUM); where many cells tie the other routes are the faster ones (RANGE, times rounded to half a mean iteration, n=93, R=211,
// B=64 494 us / 99).
constexpr int CELL_ASKED_RANGE = 48, CELL_ASKED_SUM = 112;
constexpr int CELL_IDLE = 32;             // elements of a row in one cell that cannot matter, from which on the row is taken to stand still (one timestamp
                                          // everywhere, n=1024, R=1024, B=8 511 us / 58 on the filter route: one thread goes through them)
constexpr float CELL_OFF = 64.f;          // RANGE: elements by which a row's middle is off its estimate, root mean square, from which on the rows are far from
                                          // arithmetic: what the estimate misses is read by one thread, eight elements after the other (gaps with a power-law
                                          // tail, n=1024, R=1024, B=8 305 us / 60 on the filter route, bursts of iterations 301 / 70; but iterations that grow
                                          // fivefold, R=256 and 43 off, n=128, B=256 65 / 284)
constexpr int CELL_FEW = 8;               // so many cells are asked for in any case
constexpr int CELL_SLACK = 4;             // elements by which a row may be off its estimate before a further piece is read
constexpr int GUARD_BINS = 64;            // rows by their span, eight bins to a factor of two below the longest
constexpr float GUARD_IRREGULAR = 32.f;   // bins by which more rows are looked through, to a unit of their gaps' relative deviation above 0.1
constexpr float RANGE_CELLS = 100.f;      // RANGE: cells to the longest mean iteration
constexpr float SUM_WIDTH = 0.12f;        // SUM: n cell widths against the spread of the wait over time (see k_cells)

// ------------------------------------------------------------------------------ rows
// Relative times of an instance's rows, 32 bits: elements before the first are at time 0 (before everything), those behind
// the last infinite.  in(): one element known to exist.  eight(): T[0] = element i - 1, T[k] = element i + k - 1, with i as
// given by align() (a 32-byte boundary of memory): two 32-byte loads and a single one, all under way together.
template <class SRC> struct RowReader;
template <> struct RowReader<MatBatch> {
    const int64_t *inst; int R; uint32_t tminlo;
    __device__ __forceinline__ RowReader(const MatBatch &s, int b, int n, int R_, int64_t tmin)
        : inst(s.ts + (size_t)b * n * R_), R(R_), tminlo((uint32_t)(uint64_t)tmin - 1u) {}
    __device__ __forceinline__ uint32_t in(int row, int i) const { return (uint32_t)(uint64_t)ldg64(inst + (size_t)row * R + i) - tminlo; }
    __device__ __forceinline__ void eight(int row, int i, uint32_t (&T)[9]) const {
        const int64_t *p = inst + (size_t)row * R + i;
        uint64_t v[9];
        v[0] = tminlo;
        if (i > 0) v[0] = (uint64_t)ldg64(p - 1);
        if (i >= 0 && i + 8 <= R) {
            asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[1]), "=l"(v[2]), "=l"(v[3]), "=l"(v[4]) : "l"(p));
            asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[5]), "=l"(v[6]), "=l"(v[7]), "=l"(v[8]) : "l"(p + 4));
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                v[k + 1] = i + k < 0 ? (uint64_t)tminlo : (uint64_t)tminlo - 1u;
                if ((unsigned)(i + k) < (unsigned)R) v[k + 1] = (uint64_t)ldg64(p + k);
            }
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) T[k] = (uint32_t)v[k] - tminlo;
    }
    __device__ __forceinline__ int align(int row, int i) const { return i - (int)(((uintptr_t)(inst + (size_t)row * R + i) >> 3) & 3u); }
    __device__ __forceinline__ void prefetch(int row, int i) const {
        const int64_t *p = inst + (size_t)row * R + i;
        if (i >= 0 && i + 8 <= R) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 4));
        }
    }
};
template <> struct RowReader<AriBatch> {
    const int64_t *last, *iv; int R; uint32_t tminlo;
    __device__ __forceinline__ RowReader(const AriBatch &s, int b, int n, int R_, int64_t tmin)
        : last(s.last + (size_t)b * n), iv(s.iv + (size_t)b * n), R(R_), tminlo((uint32_t)(uint64_t)tmin - 1u) {}
    __device__ __forceinline__ uint32_t in(int row, int i) const {
        return (uint32_t)(uint64_t)ldg64(last + row) - tminlo + (uint32_t)(i + 1) * (uint32_t)(uint64_t)ldg64(iv + row);
    }
    __device__ __forceinline__ void eight(int row, int i, uint32_t (&T)[9]) const {
        const uint32_t v = (uint32_t)(uint64_t)ldg64(iv + row);
        uint32_t t = in(row, i - 1);
#pragma unroll
        for (int k = 0; k < 9; ++k, t += v) T[k] = i + k - 1 < 0 ? 0u : i + k - 1 < R ? t : INF32;
    }
    __device__ __forceinline__ int align(int, int i) const { return i; }
    __device__ __forceinline__ void prefetch(int, int) const {}
};
template <class RD>
__device__ __forceinline__ uint32_t element(const RD &rd, int row, int i) { return i < 0 ? 0u : i < rd.R ? rd.in(row, i) : INF32; }

// The elements of up to 32 rows (a row a lane: `row`, its first and last element) that the time range [a, b) needs, by the
// whole warp.  A row is taken in pieces of eight elements, a piece a thread; the pieces of the warp's rows are dealt out to
// its lanes one after the other, whatever their rows.  (A warp on one row at a time, two elements a lane, spends its
// instructions on lanes outside the range and on bookkeeping: n=1024, R=1024, B=64 80 us instead of 41 for this pass.)
// Rows are close to arithmetic, so which pieces a row needs is estimated from its ends; where the estimate falls short on
// either side the thread of the first or last piece reads on.  act(T) gets nine consecutive times, eight pairs of
// neighbours: every pair with one of its elements in the range, and the pair that straddles a, comes exactly once; others
// may come.  The caller leaves out rows without an element in the range.  Returns the number of pieces.
template <class RD, class ACT>
__device__ __forceinline__ int stream_rows(const RD &rd, int R, int row, bool have, uint32_t e0, uint32_t eR, uint32_t a, uint32_t b, ACT act) {
    const int lane = threadIdx.x & 31;
    int s0 = 0, np = 0;
    if (have) {
        const float f = eR > e0 ? (float)(R - 1) / (float)(eR - e0) : 0.f;
        if (a > e0) s0 = max(0, min((int)((float)(a - e0) * f) - CELL_SLACK, R - 1));
        s0 = rd.align(row, s0);
        const int last = b > eR ? R : min((int)((float)(b - e0) * f) + 1 + CELL_SLACK, R);
        np = max(1, (last - s0 + 8) >> 3);
    }
    int incl = np;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const int y = __shfl_up_sync(FULL, incl, d); if (lane >= d) incl += y; }
    const int total = __shfl_sync(FULL, incl, 31);
    const int sb = s0 - 8 * (incl - np);                          // piece q of the warp starts at element sb + 8 q of its row
    // the lane's piece of the 32 from q0 on: its row, its first element, whether it is its row's first or last one
    int r = 0, ns = 0;
    unsigned edge = 0;
    auto assign = [&](int q0) {
        const int q = min(q0 + lane, total - 1);
        int j = 0;                                                // the lane whose row piece q belongs to
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) if (__shfl_sync(FULL, incl, j + d - 1) <= q) j += d;
        const int end = __shfl_sync(FULL, incl, j), first = end - __shfl_sync(FULL, np, j);
        r = __shfl_sync(FULL, row, j);
        ns = __shfl_sync(FULL, sb, j) + 8 * q;
        edge = (q == first ? 1u : 0u) | (q == end - 1 ? 2u : 0u);
    };
    if (total > 0) assign(0);
#pragma unroll 1
    for (int q0 = 0; q0 < total; q0 += 32) {
        const bool mine = q0 + lane < total;
        const int row_q = r;
        int s = ns;
        int back = (edge & 1u) ? s : 0, fwd = (edge & 2u) ? s + 8 : R + 1;     // where the row may have to be read on
        if (q0 + 32 < total) {                                    // the next piece on its way to the L2 while this one is worked on
            assign(q0 + 32);
            if (q0 + 32 + lane < total) rd.prefetch(r, ns);
        }
        if (mine) {
#pragma unroll 1
            for (;;) {
                uint32_t T[9];
                rd.eight(row_q, s, T);
                act(T);
                if (s <= back && (s <= 0 || T[0] < a)) back = 0;  // the row's start of the range is covered
                if (s + 8 >= fwd && T[8] >= b) fwd = R + 1;       // ... and its end
                if (back > 0) s = back = back - 8;
                else if (fwd <= R) { s = fwd; fwd += 8; }
                else break;
            }
        }
    }
    return total;
}

// Index of a row's first element at or after time t, by one thread: windows of eight elements (and the one before them), the
// first around the place that the row's ends suggest, the next ones where the mean interval puts t from the end of the
// window nearest to it; then doubling steps and bisection.
template <class RD>
__device__ __noinline__ int first_at_or_after(const RD rd, int row, int R, uint32_t t, uint32_t e0, uint32_t eR) {
    if (t <= e0) return 0;
    if (t > eR) return R;
    const float inv = (float)(R - 1) / (float)(eR - e0);          // e0 < t <= eR
    int lo = 0, hi = R - 1;                                       // element lo is before t, element hi is not
    int g = (int)((float)(t - e0) * inv);
#pragma unroll 1
    for (int it = 0; it < 4; ++it) {
        const int s = rd.align(row, min(max(g - 2, 0), R - 1));
        uint32_t T[9];
        rd.eight(row, s, T);
        int c = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k) c += T[k] < t ? 1 : 0;        // sorted: the first c of them
        if (c > 0 && c < 9) return s - 1 + c;
        if (c == 0) { hi = min(hi, s - 1); g = s - 1 - (int)min((float)(T[0] - t) * inv, (float)R); }
        else { lo = max(lo, s + 7); g = s + 8 + (int)min((float)(t - T[8]) * inv, (float)R); }
        g = min(max(g, lo), hi);
    }
    const bool up = g - lo < hi - g;
#pragma unroll 1
    for (int step = 8; hi - lo > 1; step <<= 1) {
        const int q = up ? min(lo + step, hi - 1) : max(hi - step, lo + 1);
        if (rd.in(row, q) < t) { lo = q; if (!up) break; } else { hi = q; if (up) break; }
    }
#pragma unroll 1
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (rd.in(row, mid) < t) lo = mid; else hi = mid;
    }
    return hi;
}

// Whether one of `rows` consecutive rows decreases somewhere: a warp a row, four elements a lane and step.
static __device__ bool rows_unsorted(const int64_t *ts, int rows, int R) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    bool bad = false;
#pragma unroll 1
    for (int r = warp; r < rows; r += nw) {
        const int64_t *row = ts + (size_t)r * R;
        int64_t tail = INT64_MIN;
#pragma unroll 1
        for (int i0 = 0; i0 < R; i0 += 128) {
            int64_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) { const int i = i0 + 32 * k + lane; v[k] = i < R ? ldg64(row + i) : INT64_MAX; }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                int64_t p = (int64_t)shfl_up((uint64_t)v[k], 1);
                if (lane == 0) p = tail;
                bad |= v[k] < p;
                tail = (int64_t)shfl_idx((uint64_t)v[k], 31);
            }
        }
    }
    return bad;
}

// ------------------------------------------------------------------------------ the search
struct CellParams {
    int n, R, B;
    int cap;                         // cells a CTA has room for (a multiple of 128)
    int rpc;                         // rows of a CTA when rows are asked
    int check_sorted;                // every row is read once to see that it does not decrease
    InstMeta *meta;
    uint32_t epoch;                  // number of the call: a word of `flags` is raised when it holds this
    uint32_t *flags;                 // [1] some instance needs the segment sweep, [2] some instance's outputs are missing,
                                     // [3] the calls to come should rather not take this route, [4], [5] grid_barrier
    int32_t *idx; int64_t *barrier; int64_t *wait; int32_t *status;
};

struct CellShared {
    // from every CTA of the cluster (each array is written by the others before one cluster barrier and read after it, so no
    // two exchanges share one): minima and maxima of its rows' ends; whether one of its rows decreases; SUM its rows' wait at
    // the sample time; the key of its best cell, and G or S at its start
    unsigned long long ex[4][CELL_CLUSTER];
    float exi[CELL_CLUSTER];                      // RANGE: how irregular its rows are (sum over a few of them, see k_cells)
    unsigned long long exc[CELL_CLUSTER], exs[CELL_CLUSTER], exv[CELL_CLUSTER], exb[CELL_CLUSTER];
    unsigned long long red[4][32];
    unsigned long long acc, total, key, kbase;
    uint32_t hist[GUARD_BINS];
    float span;                                   // RANGE: rows of at least this span are guards
    unsigned int pieces;                          // RANGE: pieces of eight elements that the slice took
    unsigned long long later;                     // RANGE: about how many timestamps of the other rows lie in the range
    // the cells to evaluate (in every CTA), and the order in which that is done
    uint32_t cell[CELL_ALIVE];
    uint64_t base[CELL_ALIVE];                    // RANGE: a lower bound of G at the cell's start, SUM: S there
    uint64_t lb[CELL_ALIVE];                      // lower bound of the objective in the cell
    unsigned short order[CELL_ALIVE];
    unsigned int ncells;
    uint32_t gmaxl[CELL_BATCH], gminl[CELL_BATCH];   // RANGE: latest and earliest of the own rows' first elements at or after the cell's start
    // in the first CTA: what the rows answered
    uint32_t gmax[CELL_BATCH], gmin[CELL_BATCH];  // RANGE: ... of all rows'
    uint64_t node[CELL_NODES];                    // the elements in the cells: time << 32 | RANGE the row's next element, SUM the element less the row's previous one
    unsigned int nnodes;
    int asked;                                    // (in every CTA) cells evaluated, see CELL_ASKED_*
    uint64_t tmp[34];
    unsigned int sstatus;
    unsigned int slow;                            // (in every CTA) rows far from arithmetic, or standing still
    SegResult best;                               // (in every CTA) the smallest objective so far
};

// A cell's last time; `limit` is where the timeline (or a CTA's slice of it) ends.  Formed from what is left of it behind the
// cell's start: start + width would pass 2^32 in the last cell of a timeline that ends just below.
__device__ __forceinline__ uint32_t cell_end(uint32_t start, uint32_t shift, uint32_t limit) {
    return start + min((1u << shift) - 1u, limit - 1u - start);
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(FULL, x, d);
    return x;
}

// The exact minimum over `ns` listed cells, from sh.order[from] on (in every CTA of the cluster the same): every CTA asks
// its rows, the first one evaluates and hands the result to the others.  Every thread of the cluster calls; two cluster
// barriers.  False: more elements than there is room for.
template <int OBJ, class RD>
__device__ __noinline__ bool evaluate_cells(CellShared &sh, int from, int ns, const RD rd, const uint2 *ends, int n, int R, int r0, int nrows,
                                            uint32_t lo, uint32_t hi, uint32_t shift) {
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x, nt = blockDim.x, G = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    CellShared &ld = *cl.map_shared_rank(&sh, 0);
#pragma unroll 1
    for (int q = tid; q < ns * nrows; q += nt) {                  // a (cell, row) pair a thread
        const int k = q / nrows, p = q - k * nrows;
        const int x = sh.order[from + k];
        const uint32_t a = lo + (sh.cell[x] << shift);
        const uint32_t e = cell_end(a, shift, hi);
        const uint64_t base = sh.base[x];
        const uint2 en = ends[r0 + p];
        int i = first_at_or_after(rd, r0 + p, R, a, en.x, en.y);
        uint32_t T = element(rd, r0 + p, i), pv = OBJ == ZL_OBJ_SUM ? element(rd, r0 + p, i - 1) : 0u;
        if (OBJ == ZL_OBJ_RANGE) {
            if (T > sh.gmaxl[k]) atomicMax(&sh.gmaxl[k], T);
            if (T < sh.gminl[k]) atomicMin(&sh.gminl[k], T);
        }
        int idle = 0;
#pragma unroll 1
        for (; i < R && T <= e; ++i) {
            const uint32_t nx = element(rd, r0 + p, i + 1);
            const uint32_t pay = OBJ == ZL_OBJ_RANGE ? nx : T - pv;
            // (RANGE: an element that does not raise the running maximum cannot matter)
            if (OBJ == ZL_OBJ_RANGE ? (uint64_t)nx > base : pay != 0u) {
                const unsigned pos = atomicAdd(&ld.nnodes, 1u);
                if (pos < CELL_NODES) ld.node[pos] = ((uint64_t)T << 32) | pay;
            } else if (++idle == CELL_IDLE) {
                sh.slow = 1;
            }
            pv = T; T = nx;
        }
    }
    if (OBJ == ZL_OBJ_RANGE) {
        __syncthreads();
        if (tid < ns) {
            atomicMax(&ld.gmax[tid], sh.gmaxl[tid]); atomicMin(&ld.gmin[tid], sh.gminl[tid]);
            sh.gmaxl[tid] = 0; sh.gminl[tid] = INF32;
        }
    }
    cl.sync();
    if (rank == 0) {
        const int m = (int)sh.nnodes;
        uint64_t bd = ~0ull, bt = ~0ull;
        if (m <= CELL_NODES) {
#pragma unroll 1
            for (int i = tid; i < m; i += nt) {
                const uint32_t T = (uint32_t)(sh.node[i] >> 32), c = (T - lo) >> shift;
                uint64_t v = 0;
#pragma unroll 1
                for (int k = 0; k < ns; ++k) {
                    const int x = sh.order[from + k];
                    if (sh.cell[x] == c) v = OBJ == ZL_OBJ_RANGE ? (uint64_t)sh.gmax[k] : sh.base[x];
                }
#pragma unroll 4
                for (int k = 0; k < m; ++k) {
                    const uint32_t t = (uint32_t)(sh.node[k] >> 32), pay = (uint32_t)sh.node[k];
                    if ((t - lo) >> shift != c) continue;
                    if (OBJ == ZL_OBJ_RANGE) { if (t < T) v = max(v, (uint64_t)pay); }       // max(Z): latest next of the earlier elements
                    else if (t <= T) v += pay;                                               // S: every delta up to T
                }
                const uint64_t d = OBJ == ZL_OBJ_SUM ? (uint64_t)n * T - v : v >= INF32 ? ~0ull : v - T;
                if (d != ~0ull && (d < bd || (d == bd && (uint64_t)T < bt))) { bd = d; bt = T; }
            }
            if (OBJ == ZL_OBJ_RANGE && tid < ns && sh.gmax[tid] != INF32 && sh.gmin[tid] < hi) {
                // the first element at or after the cell's start, wherever it is
                const uint64_t d = (uint64_t)(sh.gmax[tid] - sh.gmin[tid]), t = sh.gmin[tid];
                if (d < bd || (d == bd && t < bt)) { bd = d; bt = t; }
            }
        }
        if (tid == 0 && (sh.best.d < bd || (sh.best.d == bd && sh.best.t < bt))) { bd = sh.best.d; bt = sh.best.t; }
        __syncthreads();
        block_best_to_result(bd, bt, ZL_OK, sh.tmp, &sh.sstatus, sh.best);
        if (tid == 0) { if (m > CELL_NODES) sh.best.valid = 0; sh.nnodes = 0; }
        if (tid < CELL_BATCH) { sh.gmax[tid] = 0; sh.gmin[tid] = INF32; }
        __syncthreads();
        const SegResult r = sh.best;
        if (tid > 0 && tid < G) cl.map_shared_rank(&sh, tid)->best = r;
    }
    cl.sync();
    return sh.best.valid != 0;
}

// Dynamic shared memory: the slice's cells [cap + 4] u32 | rows' first and last element, relative [n] uint2 | SUM: per 128
// cells the scan before them and the smallest lower bound among them [cap / 128] two u64.
template <int OBJ, class SRC>
__global__ void __launch_bounds__(1024, 1) k_cells(const SRC src, const CellParams P) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ CellShared sh;
    cg::cluster_group cl = cg::this_cluster();
    const int b = blockIdx.y, rank = blockIdx.x, G = gridDim.x;
    // A CTA's shared memory may be written by the others only once it runs: everybody says so here, and waits for the rest
    // with the columns read, before the first store into another CTA.
    if (G > 1) cl.barrier_arrive();
    grid_dep_wait();
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int n = P.n, R = P.R;
    uint32_t *cell = (uint32_t *)smem;
    uint2 *ends = (uint2 *)(cell + P.cap + 4);
    uint64_t *blk_before = (uint64_t *)(ends + n), *blk_lb = blk_before + P.cap / 128;
    const int r0 = min(rank * P.rpc, n), nrows = min(P.rpc, n - r0);
    if (b == 0 && rank == 0 && tid < 2) P.flags[4 + tid] = 0;      // (used by the last kernel only)
    // ---- columns of the own rows; everybody gets everybody's minima and maxima and the low words of the rows' ends
    {
        const typename SRC::Rows rows = src.inst(b, n, R);
        uint64_t q[4] = {~0ull, 0, ~0ull, 0};                     // order-preserving unsigned images of int64
        float irr = 0.f;
        const int step = (n + 31) / 32;
#pragma unroll 1
        for (int p = tid; p < nrows; p += nt) {
            const auto row = rows.row(r0 + p);
            const int64_t x = row.at(0), y = row.at(R - 1);
            if (OBJ == ZL_OBJ_RANGE && R > 2 && (r0 + p) % step == 0) {
                // RANGE, a few dozen rows: how far the row's middle element is from where a row of equal gaps has it, in gaps: after h of R - 1
                // gaps with a standard deviation of s (in gaps) that is s * sqrt(h * (R - 1 - h) / (R - 1)) on average
                const int h = (R - 1) / 2;
                const float span = (float)(y - x), off = (float)(row.at(h) - x) * (float)(R - 1) - span * (float)h;
                if (span > 0.f) irr += off * off / (span * span) * ((float)(R - 1) / ((float)h * (float)(R - 1 - h)));
            }
            const uint64_t ux = (uint64_t)x ^ (1ull << 63), uy = (uint64_t)y ^ (1ull << 63);
            q[0] = min(q[0], ux); q[1] = max(q[1], ux); q[2] = min(q[2], uy); q[3] = max(q[3], uy);
            ends[r0 + p] = make_uint2((uint32_t)(uint64_t)x, (uint32_t)(uint64_t)y);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q[k] = (k & 1) ? warp_reduce(q[k], OpMax()) : warp_reduce(q[k], OpMin());
            if (lane == 0) sh.red[k][warp] = q[k];
        }
        if (OBJ == ZL_OBJ_RANGE) {
            irr = warp_sum(irr);
            if (lane == 0) sh.tmp[warp] = (uint64_t)__float_as_uint(irr);
        }
        if (tid == 0) {
            sh.acc = 0; sh.total = 0; sh.key = ~0ull; sh.ncells = 0; sh.nnodes = 0; sh.sstatus = 0; sh.later = 0; sh.pieces = 0; sh.slow = 0; sh.asked = 0;
            sh.best.d = sh.best.t = ~0ull; sh.best.valid = 0; sh.best.status = 0;
        }
        if (tid < CELL_BATCH) { sh.gmax[tid] = sh.gmaxl[tid] = 0; sh.gmin[tid] = sh.gminl[tid] = INF32; }
#pragma unroll 1
        for (int k = tid; k < GUARD_BINS; k += nt) sh.hist[k] = 0;
        __syncthreads();
        if (G > 1) {
            cl.barrier_wait();
#pragma unroll 1
            for (int r = 0; r < G; ++r) {
                if (r == rank) continue;
                uint2 *to = cl.map_shared_rank(ends, r);
#pragma unroll 1
                for (int p = tid; p < nrows; p += nt) to[r0 + p] = ends[r0 + p];
            }
        }
        if (tid < 4 * G) {
            const int k = tid & 3, r = tid >> 2;
            unsigned long long v = sh.red[k][0];
#pragma unroll 1
            for (int w = 1; w < nw; ++w) v = (k & 1) ? max(v, sh.red[k][w]) : min(v, sh.red[k][w]);
            cl.map_shared_rank(&sh, r)->ex[k][rank] = v;
            if (OBJ == ZL_OBJ_RANGE && k == 0) {
                float v = 0.f;
#pragma unroll 1
                for (int w = 0; w < nw; ++w) v += __uint_as_float((uint32_t)sh.tmp[w]);
                cl.map_shared_rank(&sh, r)->exi[rank] = v;
            }
        }
    }
#pragma unroll 1
    for (int c = tid; c <= P.cap / 4; c += nt) reinterpret_cast<uint4 *>(cell)[c] = make_uint4(0, 0, 0, 0);
    if constexpr (std::is_same<SRC, MatBatch>::value) if (P.check_sorted) {
        const bool bad = rows_unsorted(src.ts + ((size_t)b * n + r0) * R, nrows, R);
        const int any = __syncthreads_or(bad);
        if (tid < G) cl.map_shared_rank(&sh, tid)->exc[rank] = any ? 1ull : 0ull;
    }
    cl.sync();
    InstMeta M;
    {
        uint64_t q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q[k] = sh.ex[k][0];
#pragma unroll 1
            for (int r = 1; r < G; ++r) q[k] = (k & 1) ? max(q[k], (uint64_t)sh.ex[k][r]) : min(q[k], (uint64_t)sh.ex[k][r]);
        }
        const int64_t tmin = (int64_t)(q[0] ^ (1ull << 63)), t0 = (int64_t)(q[1] ^ (1ull << 63));
        const int64_t lmin = (int64_t)(q[2] ^ (1ull << 63)), tmax = (int64_t)(q[3] ^ (1ull << 63));
        M.tmin = tmin; M.status = ZL_OK;
        M.cscale = 0; M.fscale = 0; M.count = 0; M.count2 = 0; M.overflow = 0; M.dmin = 0;
        if (tmin < 0 || tmax >= VALUE_LIMIT || tmax < tmin || lmin < tmin) {
            M.status = ZL_ERR_INVALID_ARG;                        // outside [0, 2^62), or first/last columns out of order
            M.t0 = M.lmin = M.tend = 1; M.use32 = 1;
        } else {
            M.t0 = (uint64_t)(t0 - tmin) + 1;
            M.lmin = (uint64_t)(lmin - tmin) + 1;
            M.tend = (uint64_t)(tmax - tmin) + 1;
            M.use32 = M.tend < 0xfffffffeull;
            if (OBJ == ZL_OBJ_SUM && M.tend > (uint64_t)INT64_MAX / (uint64_t)n) M.status = ZL_ERR_UNSUPPORTED;
        }
        if (P.check_sorted && M.status == ZL_OK) {
#pragma unroll 1
            for (int r = 0; r < G; ++r) if (sh.exc[r]) M.status = ZL_ERR_UNSORTED;
        }
        M.cscale = M.status == ZL_OK && M.use32 ? 1u : 0u;
    }
    if (!M.cscale) {                                              // the same in the whole cluster
        if (rank == 0 && tid == 0) {
            P.meta[b] = M;
            P.flags[2] = P.epoch;                                 // the last kernel writes this instance's outputs
            if (M.status == ZL_OK) P.flags[1] = P.flags[3] = P.epoch;
        }
        return;
    }
    const RowReader<SRC> rd(src, b, n, R, M.tmin);
    const uint32_t t0 = (uint32_t)M.t0, lmin = (uint32_t)M.lmin, tend = (uint32_t)M.tend, tminlo = (uint32_t)(uint64_t)M.tmin - 1u;
    uint32_t lo = 1, hi = lmin + 1, shift;
    uint64_t ub = ~0ull;                                          // SUM: a wait that is attained
    float width;                                                  // what a cell may span, in time units
    {
        uint32_t longest = 0;
#pragma unroll 1
        for (int p = tid; p < n; p += nt) {
            uint2 e = ends[p];
            e.x -= tminlo; e.y -= tminlo;
            ends[p] = e;
            longest = max(longest, e.y - e.x);
        }
        longest = __reduce_max_sync(FULL, longest);
        if (lane == 0) sh.red[0][warp] = longest;
        __syncthreads();
        longest = (uint32_t)sh.red[0][0];
#pragma unroll 1
        for (int w = 1; w < nw; ++w) longest = max(longest, (uint32_t)sh.red[0][w]);
        if (OBJ == ZL_OBJ_RANGE) {
            // Guards: the rows that can set G near the optimum.  At a random time row i's next element is uniform in its mean
            // gap m_i away, so all are within x with probability prod(x / m_i) over the rows with m_i > x; the smallest d of
            // about N = n * R tries is the x where sum(log(m_i / x)) reaches log(N), and rows with gaps shorter than that
            // hardly matter.  With the rows counted by the logarithm of their span that is a prefix sum of a prefix sum.  Rows
            // a bin shorter are taken along, and more of them where single gaps are much longer than the row's mean.  (A fifth
            // to a half of the rows on the workloads at hand.  A fixed fifth leaves dozens of cells where single gaps are
            // long: n=1024, R=1024, B=64 87 us; a fixed half costs n=128, R=256, B=1024 68 us instead of 53.)
            const int top = __float_as_int((float)longest) >> 20;
#pragma unroll 1
            for (int p = tid; p < n; p += nt) {
                const uint2 e = ends[p];
                atomicAdd(&sh.hist[min(GUARD_BINS - 1, top - (__float_as_int((float)(e.y - e.x)) >> 20))], 1u);
            }
            __syncthreads();
            if (warp == 0) {
                const uint32_t x0 = sh.hist[2 * lane], x1 = sh.hist[2 * lane + 1];
                uint32_t inc = x0 + x1;                           // rows in the bins up to the lane's second one
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, inc, d); if (lane >= d) inc += y; }
                const uint32_t n0 = inc - x1, n1 = inc;           // rows up to bin 2 lane, 2 lane + 1
                uint32_t dep = n0 + n1;                           // sum of these over the bins: (bin - own bin) over the rows, from the next bin on
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, dep, d); if (lane >= d) dep += y; }
                const uint32_t d0 = dep - n0 - n1, d1 = dep - n1; // that sum at bin 2 lane, 2 lane + 1
                const uint32_t tries = (uint32_t)(8.f * log2f((float)n * (float)R)), least = (uint32_t)min(n, 8);
                int k = __reduce_min_sync(FULL, d0 >= tries ? 2 * lane : d1 >= tries ? 2 * lane + 1 : GUARD_BINS);
                float irr = 0.f;
#pragma unroll 1
                for (int r = 0; r < G; ++r) irr += sh.exi[r];
                const float dev = sqrtf(irr / (float)((n + (n + 31) / 32 - 1) / ((n + 31) / 32)));
                if (lane == 0 && dev * sqrtf((float)R) > 2.f * CELL_OFF) sh.slow = 1;      // (dev * sqrt(R) / 2 elements in the middle)
                k += 1 + (int)(GUARD_IRREGULAR * max(0.f, min(1.f, dev) - 0.1f));
                k = max(k, __reduce_min_sync(FULL, n0 >= least ? 2 * lane : n1 >= least ? 2 * lane + 1 : GUARD_BINS));
                if (lane == 0) sh.span = k >= min(GUARD_BINS - 1, top) ? 0.f : __int_as_float((top - k) << 20);
            }
            __syncthreads();
            const float span = sh.span;
            float el = 0.f;
#pragma unroll 1
            for (int p = tid; p < n; p += nt) {
                const float w = (float)(ends[p].y - ends[p].x);
                if (w < span) el += min(1.f, (float)(lmin - min(lmin, ends[p].x)) / w) * (float)R;
            }
            el = warp_sum(el);
            if (lane == 0) atomicAdd(&sh.later, (unsigned long long)el);
            width = R > 1 ? (float)longest / ((float)(R - 1) * RANGE_CELLS) : 0.f;
        } else {
            // the wait at one time between the last worker's start and the first row's end
            const uint32_t lm = max(lmin, t0), t = t0 + (lm - t0) / 2;
            uint64_t acc = 0;
#pragma unroll 1
            for (int p = tid; p < nrows; p += nt) {
                const uint2 e = ends[r0 + p];
                const int i = first_at_or_after(rd, r0 + p, R, t + 1u, e.x, e.y);
                acc += t - rd.in(r0 + p, max(0, i - 1));
            }
            acc = warp_reduce(acc, OpAdd());
            if (lane == 0) atomicAdd(&sh.acc, (unsigned long long)acc);
            __syncthreads();
            if (tid < G) cl.map_shared_rank(&sh, tid)->exs[rank] = sh.acc;
            cl.sync();
            ub = 0;
#pragma unroll 1
            for (int r = 0; r < G; ++r) ub += sh.exs[r];
            // times past lm at which the exhausted rows alone wait longer than that are left out: the first of 32 trial times
            // where they do (closer together near lm), then the first of 32 more between that one and the one before it
            unsigned long long *es = (unsigned long long *)sh.node;              // (64 words, not in use yet)
            if (tid < 64) es[tid] = 0;
            if (tid == 0) sh.acc = 0;
            uint32_t below = lm, stop = lm + (uint32_t)min(ub, (uint64_t)(tend - lm));
#pragma unroll 1
            for (int part = 0; part < 2; ++part, es += 32) {
                __syncthreads();
                const uint64_t k = part ? 32ull * (lane + 1) : (uint64_t)((lane + 1) * (lane + 1));
                const uint32_t trial = below + (uint32_t)(((uint64_t)(stop - below) * k) >> 10);
                uint64_t e = 0;
#pragma unroll 1
                for (int p = warp; p < n; p += nw) { const uint32_t last = ends[p].y; e += trial > last ? trial - last : 0u; }
                atomicAdd(&es[lane], (unsigned long long)e);
                __syncthreads();
                const unsigned over = __ballot_sync(FULL, es[lane] > ub);
                const int first = over ? __ffs(over) - 1 : 32;
                const uint32_t at = __shfl_sync(FULL, trial, min(first, 31)), before = __shfl_sync(FULL, trial, max(first - 1, 0));
                if (first > 0) below = before;
                if (first < 32) stop = at;
                else { stop = part ? stop : tend; below = stop; }
            }
            lo = t0;
            hi = max(lo, min(stop, tend)) + 1u;
            // n cell widths are the looseness of a cell's bounds; the wait itself spreads over time by about sqrt(n) times
            // 0.29 iterations, an iteration being about twice the mean wait of a worker.  (n=17, R=700, B=20: half the factor
            // 73 us, twice the factor 840, with six instances left over; n=32, R=400, B=20 41, 39 and 68.)
            width = SUM_WIDTH * (float)ub / ((float)n * sqrtf((float)n));
            __syncthreads();                                      // es has been read
        }
    }
    shift = width >= 2.f ? (uint32_t)min(31, (__float_as_int(width) >> 23) - 127) : 0u;
    while (((hi - lo - 1u) >> shift) >= (uint32_t)(G * P.cap)) ++shift;
    const uint32_t ncells = ((hi - lo - 1u) >> shift) + 1u;
    const uint32_t per = ((ncells + G - 1) / G + 3u) & ~3u;       // cells of a CTA (cap is a multiple of 128, so they fit)
    const uint32_t c0 = min((uint32_t)rank * per, ncells), c1 = min(c0 + per, ncells);
    const int m = (int)(c1 - c0), nblk = (m + 127) >> 7;
    const uint32_t a = lo + (c0 << shift), bnd = c1 == ncells ? hi : lo + (c1 << shift);
    bool fits = true;
    uint32_t gap = 0;                                             // RANGE: no cell's bound is below this
    uint64_t low = 0;                                             // cells with keys up to this have been evaluated
    int stage = 0, streamed = -1;                                 // RANGE: 0 the guards, 1 (seldom) the other rows too
#pragma unroll 1
    for (int round = 0;; ++round) {                               // a round: the most promising cell is evaluated, the rest counted
        // ---- the rows' elements in the slice
        if (m > 0 && streamed != stage) {
            uint64_t carry = 0, total = 0;                        // SUM: the rows' last elements before a, and all deltas in the slice
            const uint32_t w = bnd - a;
#pragma unroll 1
            for (int base = warp; base < n; base += 32 * nw) {    // warp w takes rows w, w + nw, ..., a row a lane
                const int row = base + lane * nw;
                uint2 e = make_uint2(0u, 0u);
                bool have = row < n;
                if (have) {
                    e = ends[row];
                    if (OBJ == ZL_OBJ_RANGE) have = ((float)(e.y - e.x) >= sh.span) == (stage == 0);
                    if (e.x >= bnd || e.y < a) {                  // no element of the row in the slice
                        if (OBJ == ZL_OBJ_SUM && have && e.y < a) carry += e.y;
                        have = false;
                    }
                }
                const int pieces = stream_rows(rd, R, row, have, e.x, e.y, a, bnd, [&](const uint32_t (&T)[9]) {
                    if (OBJ == ZL_OBJ_RANGE) {
                        // cell[k] becomes a lower bound of G at the start of cell k (before the prefix maximum): an element
                        // says that G is at least its successor for the cells after its own.  Elements before the slice
                        // count for its first cell; those in its last cell or behind it go to cell[m], which is not looked
                        // at.  A gap of at most `gap` cannot push a cell's bound, G less the cell's end, beyond that: it discards no cell.
                        uint32_t longer = 0;
#pragma unroll
                        for (int j = 0; j < 8; ++j) longer = max(longer, T[j + 1] - T[j]);
                        if (longer > gap) {
                            uint32_t k[8], v[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                k[j] = T[j] < a ? 0u : min(((T[j] - a) >> shift) + 1u, (uint32_t)m);
                                v[j] = cell[k[j]];                // all eight under way; a value gone stale costs an update
                            }
#pragma unroll
                            for (int j = 0; j < 8; ++j) if (T[j + 1] - T[j] > gap && v[j] < T[j + 1]) atomicMax(&cell[k[j]], T[j + 1]);
                        }
                    } else {
                        uint32_t in = 0, before = 0;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const uint32_t d = T[j + 1] - a, delta = T[j + 1] - T[j];
                            if (d < w) { atomicAdd(cell + (d >> shift), delta); in += delta; }
                            if (T[j] < a && T[j + 1] >= a) before = T[j];
                        }
                        total += in; carry += before;
                    }
                });
                if (OBJ == ZL_OBJ_RANGE && lane == 0) atomicAdd(&sh.pieces, (unsigned)pieces);
            }
            if (OBJ == ZL_OBJ_SUM) {
                carry = warp_reduce(carry, OpAdd());
                total = warp_reduce(total, OpAdd());
                if (lane == 0) { atomicAdd(&sh.acc, (unsigned long long)carry); atomicAdd(&sh.total, (unsigned long long)total); }
            }
        }
        streamed = stage;
        __syncthreads();
        // ---- what the sweep knows at every cell's start; a warp takes a run of 128-cell blocks, four cells a lane
        const int bpw = (nblk + nw - 1) / nw, k0 = min(warp * bpw, nblk), k1 = min(k0 + bpw, nblk);
        typedef typename std::conditional<OBJ == ZL_OBJ_RANGE, uint32_t, uint64_t>::type ST;
        {
            ST t = 0;
#pragma unroll 1
            for (int k = k0; k < k1; ++k) {
                const uint4 v = *reinterpret_cast<const uint4 *>(cell + 128 * k + 4 * lane);
                if constexpr (OBJ == ZL_OBJ_RANGE) t = max(max(t, max(v.x, v.y)), max(v.z, v.w));
                else t += (uint64_t)v.x + v.y + v.z + v.w;
            }
            if constexpr (OBJ == ZL_OBJ_RANGE) t = __reduce_max_sync(FULL, t); else t = warp_reduce(t, OpAdd());
            if (lane == 0) sh.red[0][warp] = t;
        }
        if (tid == 0) sh.key = ~0ull;
        __syncthreads();
        uint64_t key = ~0ull, kbase = 0;
        if constexpr (OBJ == ZL_OBJ_RANGE) {
            uint32_t run = t0;
#pragma unroll 1
            for (int w = 0; w < warp; ++w) run = max(run, (uint32_t)sh.red[0][w]);
#pragma unroll 1
            for (int k = k0; k < k1; ++k) {
                uint4 v = *reinterpret_cast<const uint4 *>(cell + 128 * k + 4 * lane);
                v.y = max(v.x, v.y); v.z = max(v.y, v.z); v.w = max(v.z, v.w);
                uint32_t inc = v.w;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, inc, d); if (lane >= d) inc = max(inc, y); }
                uint32_t before = __shfl_up_sync(FULL, inc, 1);
                before = lane ? max(run, before) : run;
                v.x = max(v.x, before); v.y = max(v.y, before); v.z = max(v.z, before); v.w = max(v.w, before);
                *reinterpret_cast<uint4 *>(cell + 128 * k + 4 * lane) = v;
                run = max(run, __shfl_sync(FULL, inc, 31));
                // the most promising cell: the smallest G(start) - end.  (The optimum lies where G is about to rise.)
                const uint32_t g[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 128 * k + 4 * lane + j;
                    const uint32_t end = cell_end(a + ((uint32_t)c << shift), shift, bnd);
                    const uint64_t q = (uint64_t)(g[j] > end ? g[j] - end : 0u) << 24 | (c0 + (uint32_t)c + 1u);      // never 0
                    if (c < m && g[j] != INF32 && q > low && q < key) { key = q; kbase = g[j]; }
                }
            }
        } else {
            uint64_t run = sh.acc, all = 0;
#pragma unroll 1
            for (int w = 0; w < nw; ++w) { if (w < warp) run += sh.red[0][w]; all += sh.red[0][w]; }
            const uint64_t nn = (uint64_t)n;
#pragma unroll 1
            for (int k = k0; k < k1; ++k) {
                const uint4 v = *reinterpret_cast<const uint4 *>(cell + 128 * k + 4 * lane);
                const uint64_t s1 = v.x, s2 = s1 + v.y, s3 = s2 + v.z, s4 = s3 + v.w;
                uint64_t inc = s4;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) { const uint64_t y = shfl_up(inc, d); if (lane >= d) inc += y; }
                const uint64_t before = run + inc - s4;
                const uint64_t S[4] = {before + s1, before + s2, before + s3, before + s4};
                const uint32_t dv[4] = {v.x, v.y, v.z, v.w};
                uint64_t lbm = ~0ull;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 128 * k + 4 * lane + j;
                    if (dv[j] != 0u) {
                        const uint32_t start = a + ((uint32_t)c << shift), end = cell_end(start, shift, bnd);
                        const uint64_t u = nn * end - S[j], l = nn * start > S[j] ? nn * start - S[j] : 0ull;
                        lbm = min(lbm, l);
                        const uint64_t q = min(u, (uint64_t)0xffffffffffull) << 24 | (c0 + (uint32_t)c + 1u);
                        if (q > low && q < key) { key = q; kbase = S[j] - dv[j]; }
                    }
                }
                lbm = warp_reduce(lbm, OpMin());
                if (lane == 0) { blk_before[k] = run; blk_lb[k] = lbm; }
                run += shfl_idx(inc, 31);
            }
            // a cell's 32-bit sum wrapped around: nothing in the slice can be trusted
            if (all != sh.total) fits = false;
        }
        {
            const uint64_t mine = warp_reduce(key, OpMin());
            if (lane == 0) atomicMin(&sh.key, (unsigned long long)mine);
            __syncthreads();
            if (key != ~0ull && key == sh.key) sh.kbase = kbase;  // (keys are different)
            __syncthreads();
            if (tid < G) {
                CellShared &to = *cl.map_shared_rank(&sh, tid);
                to.exv[rank] = fits ? sh.key : 0ull;
                to.exb[rank] = sh.kbase;
            }
        }
        cl.sync();
        uint64_t best_key = sh.exv[0];
        int owner = 0;
#pragma unroll 1
        for (int r = 0; r < G; ++r) {
            fits &= sh.exv[r] != 0ull;
            if (sh.exv[r] < best_key) { best_key = sh.exv[r]; owner = r; }
        }
        if (!fits || best_key == ~0ull) { fits = false; break; }
        // ---- the most promising cell exactly
        if (OBJ == ZL_OBJ_RANGE && round == 0) gap = (uint32_t)(best_key >> 24);
        low = best_key;
        if (tid == 0) {
            sh.cell[0] = (uint32_t)(best_key & 0xffffffu) - 1u; sh.order[0] = 0;
            sh.base[0] = sh.exb[owner];
            if (rank == 0) sh.ncells = 0;
        }
        __syncthreads();
        fits = evaluate_cells<OBJ>(sh, 0, 1, rd, ends, n, R, r0, nrows, lo, hi, shift);
        if (!fits) break;
        if (tid == 0) sh.asked += 8;
        // ---- the cells that may still hold a smaller one, or the same one earlier: only cells before the best one's
        const uint64_t d = sh.best.d;
        const uint32_t cb = ((uint32_t)sh.best.t - lo) >> shift;
        const uint64_t limit = d < INF32 ? d << 24 | (cb + 1u) : ~0ull;      // RANGE: the best one's key, as of a cell whose bound is attained
        CellShared &ld = *cl.map_shared_rank(&sh, 0);
        auto keep = [&](uint32_t c, uint64_t base, uint64_t l) {
            const unsigned pos = atomicAdd(&ld.ncells, 1u);
            if (pos < CELL_ALIVE) {
                // every CTA gets the list
#pragma unroll 1
                for (int r = 0; r < G; ++r) { CellShared &to = *cl.map_shared_rank(&sh, r); to.cell[pos] = c; to.base[pos] = base; to.lb[pos] = l; }
            }
        };
        if constexpr (OBJ == ZL_OBJ_RANGE) {
#pragma unroll 1
            for (int c = 4 * tid; c < m; c += 4 * nt) {
                const uint4 v = *reinterpret_cast<const uint4 *>(cell + c);
                const uint32_t g[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t end = cell_end(a + ((uint32_t)(c + j) << shift), shift, bnd);
                    const uint64_t l = g[j] > end ? (uint64_t)(g[j] - end) : 0ull;
                    const uint64_t q = l << 24 | (c0 + (uint32_t)(c + j) + 1u);
                    if (c + j < m && q > low && q < limit) keep(c0 + (uint32_t)(c + j), g[j], l);
                }
            }
        } else {
#pragma unroll 1
            for (int k = warp; k < nblk; k += nw) {
                if (blk_lb[k] > d) continue;
                const uint4 v = *reinterpret_cast<const uint4 *>(cell + 128 * k + 4 * lane);
                const uint64_t s1 = v.x, s2 = s1 + v.y, s3 = s2 + v.z, s4 = s3 + v.w;
                uint64_t inc = s4;
#pragma unroll
                for (int q = 1; q < 32; q <<= 1) { const uint64_t y = shfl_up(inc, q); if (lane >= q) inc += y; }
                const uint64_t before = blk_before[k] + inc - s4;
                const uint64_t S[4] = {before + s1, before + s2, before + s3, before + s4};
                const uint32_t dv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t c = (uint32_t)(128 * k + 4 * lane + j);
                    if (dv[j] != 0u) {
                        const uint32_t start = a + (c << shift), end = cell_end(start, shift, bnd);
                        const uint64_t st = (uint64_t)n * start, l = st > S[j] ? st - S[j] : 0ull;
                        const uint64_t q = min((uint64_t)n * end - S[j], (uint64_t)0xffffffffffull) << 24 | (c0 + c + 1u);
                        if ((l < d || (l == d && c0 + c < cb)) && q > low) keep(c0 + c, S[j] - dv[j], l);
                    }
                }
            }
        }
        cl.sync();
        const int ns = (int)ld.ncells;
        if (ns == 0) break;
        // asking every row for each of them, or looking through the other rows first?
        if (OBJ == ZL_OBJ_RANGE && stage == 0 && sh.span > 0.f && (ns > CELL_ALIVE || (ns > CELL_FEW && (long long)ns * n * CELL_ASK > (long long)sh.later))) {
            stage = 1; low = 0;
            continue;                                             // (a cluster barrier follows before the length is touched again)
        }
        if (ns > CELL_ALIVE) {                                    // more than there is room for: the next best cell may discard them
            fits = round < CELL_ROUNDS && ns <= CELL_HOPELESS;
            if (fits) continue;
            break;
        }
#pragma unroll 1
        for (int k = tid; k < ns; k += nt) {                      // most promising first, of equal ones the earliest
            const uint64_t l = sh.lb[k];
            const uint32_t c = sh.cell[k];
            int at = 0;
#pragma unroll 1
            for (int i = 0; i < ns; ++i) at += sh.lb[i] < l || (sh.lb[i] == l && sh.cell[i] < c);
            sh.order[at] = (unsigned short)k;
        }
        __syncthreads();
        // (SUM: a cell whose bound does not exceed d nearly always has to be looked at)
        const int batch = OBJ == ZL_OBJ_SUM ? 8 : max(4, min(CELL_BATCH, 4 * nt / P.rpc));
#pragma unroll 1
        for (int from = 0; from < ns && fits; from += batch) {
            const int x = sh.order[from];
            if (sh.lb[x] > sh.best.d || (sh.lb[x] == sh.best.d && sh.cell[x] >= ((uint32_t)sh.best.t - lo) >> shift)) break;
            if (tid == 0) sh.asked += min(batch, ns - from);
            fits = evaluate_cells<OBJ>(sh, from, min(batch, ns - from), rd, ends, n, R, r0, nrows, lo, hi, shift);
        }
        break;
    }
    // Rows that the route is not made for: many evaluations, rows that stand still, RANGE rows far off their estimates or far more of
    // them in one slice than its share.  The result is as good as any, but the handle's next calls are better off elsewhere.
    if (tid == 0 && (sh.slow || sh.asked > (OBJ == ZL_OBJ_RANGE ? CELL_ASKED_RANGE : CELL_ASKED_SUM) ||
                     (OBJ == ZL_OBJ_RANGE && G > 1 && streamed == 0 && 16ll * G * ((long long)sh.pieces - 2 * n) > 3ll * n * R)))
        P.flags[3] = P.epoch;
    cl.sync();                                                    // no CTA leaves while another may still read its memory
    // (a result above the wait known to be attained means rows that are not sorted: the sweep decides)
    if (!fits || !sh.best.valid || sh.best.d > ub) {
        if (rank == 0 && tid == 0) {
            M.overflow = 1;
            P.meta[b] = M;
            P.flags[1] = P.flags[2] = P.flags[3] = P.epoch;
        }
        return;
    }
    const SegResult best = sh.best;
    const uint32_t bar = (uint32_t)best.t + (OBJ == ZL_OBJ_RANGE ? (uint32_t)best.d : 0u);      // relative
    if (rank == 0 && tid == 0) {
        P.meta[b] = M;
        P.wait[b] = (int64_t)best.d;
        P.barrier[b] = M.tmin - 1 + (int64_t)bar;
        if (P.status) P.status[b] = ZL_OK;
    }
    // ---- the indices of the own rows: the last element not after the barrier
#pragma unroll 1
    for (int p = tid; p < nrows; p += nt) {
        const uint2 e = ends[r0 + p];
        P.idx[(size_t)b * n + r0 + p] = first_at_or_after(rd, r0 + p, R, bar + 1u, e.x, e.y) - 1;
    }
}

// ------------------------------------------------------------------------------ rest
constexpr int CELL_REST_THREADS = 512;

template <int OBJ, class SRC>
__global__ void __launch_bounds__(CELL_REST_THREADS) k_cell_rest(const SRC src, const SweepParams SP, const CellParams P, FilterBufs F) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ SweepShared sh;
    const uint4 fl = __ldcg(reinterpret_cast<const uint4 *>(P.flags));
    if (F.hint && fl.w == P.epoch && blockIdx.x == 0 && threadIdx.x == 0) F.hint[1] = P.epoch; // for the host's next calls
    if (fl.y != P.epoch && fl.z != P.epoch) return;               // every instance is finished
    bool ok = true;
    if (fl.y == P.epoch) {
        sweep_items<OBJ>(SP, src, sh, smem);
        ok = grid_barrier(P.flags + 4, P.flags + 5, 1);
        if (ldcg32(P.flags + 5)) ok = false;
    }
    finalize_all(src, P.B, P.n, P.R, SP.nseg, F, SP.nres, OBJ, 1, SP.meta, SP.seg, P.idx, P.barrier, P.wait, P.status,
                 ok ? (uint32_t)ZL_OK : (uint32_t)ZL_ERR_TIMEOUT, nullptr);
}

// ------------------------------------------------------------------------------ host side
// CTAs of an instance's cluster, their threads, and the cells each has room for.
struct CellShape { int cluster, threads, cap; size_t smem; };

static CellShape cell_shape(int n, int R, int B, int objective, int num_sms) {
    CellShape s;
    // CTAs: as many as there are SMs (SUM: two an SM), each with 16 rows at least to ask; clusters of 16 only for the largest instances, of
    // which few fill the GPU.  Threads: as many as an SM holds (clusters of 16: for two CTAs an SM, or not all of eight
    // clusters find room at once), one to so many timestamps (RANGE looks through an eighth of them).
    const int most = (long long)n * R >= (1 << 22) ? CELL_CLUSTER : 8;
    const long long per_sm_ctas = objective == ZL_OBJ_RANGE ? 1 : 2;      // (SUM n=1024, R=1024, B=64: 236 us with one, 206 with two)
    s.cluster = 1;
    while (s.cluster < most && (long long)B * s.cluster * 2 <= per_sm_ctas * num_sms && n / (s.cluster * 2) >= 16) s.cluster *= 2;
    const long long ctas = (long long)B * s.cluster;
    s.threads = ctas > 4LL * num_sms ? 128 : ctas > 2LL * num_sms ? 256 : ctas > num_sms || s.cluster > 8 ? 512 : 1024;
    const int per_thread = 32 * (objective == ZL_OBJ_RANGE ? 48 : 16);
    s.threads = (int)std::min<long long>(s.threads, std::max<long long>(128, 32 * (((long long)n * R / s.cluster + per_thread - 1) / per_thread)));
    // Cells an instance can use.  RANGE: RANGE_CELLS to an iteration of the slowest row, of which there are rarely more than
    // half R before the first row runs out.  SUM: see SUM_WIDTH, 6 to 12 sqrt(n) cells an iteration.  No more than lets the
    // CTAs of the call (up to eight an SM) be resident together: they are bound by latency, not by what they move.
    double want = objective == ZL_OBJ_RANGE ? RANGE_CELLS * 0.5 * R : 12.0 * R * std::sqrt((double)n);
    want = std::max(256.0, std::min(want, (double)(1 << 18)));
    const long long per_sm = s.cluster > 8 ? 2 : std::max<long long>(1, std::min<long long>(8, (ctas + num_sms - 1) / num_sms));
    const double cell_bytes = objective == ZL_OBJ_RANGE ? 4.0 : 4.125;
    const double room = (std::min(200.0, 224.0 / (double)per_sm) * 1024 - sizeof(CellShared) - 1024 - 8.0 * n - 64) / cell_bytes;
    const int most_cells = std::max(2048, (int)room & ~127);
    s.cap = std::min(most_cells, ((int)(want / s.cluster) + 127) & ~127);
    s.cap = std::max(256, s.cap);
    s.smem = (size_t)s.cap * 4 + 16 + (size_t)n * 8 + (objective == ZL_OBJ_RANGE ? 0 : (size_t)s.cap / 8);
    return s;
}

template <int OBJ, class SRC>
static void enqueue_cells_t(const Pipeline &q, const FilterBufs &fb, const LaunchPlan &p, cudaStream_t st, cudaEvent_t *ev, const SRC &src) {
    const CellShape s = cell_shape(q.n, q.R, q.B, OBJ, q.num_sms);
    CellParams P;
    P.n = q.n; P.R = q.R; P.B = q.B;
    P.cap = s.cap; P.rpc = (q.n + s.cluster - 1) / s.cluster; P.check_sorted = (q.flags & ZL_FLAG_CHECK_SORTED) ? 1 : 0;
    P.meta = q.meta; P.flags = q.cflags; P.epoch = q.epoch;
    P.idx = q.idx; P.barrier = q.barrier; P.wait = q.wait; P.status = q.status;
    auto launch = [&](auto kernel, dim3 grid, int threads, size_t smem, int cluster, auto... args) {
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = cluster > 1 ? 2 : 1;
        cudaLaunchKernelEx(&cfg, kernel, args...);
    };
    if (q.cells != 3) launch(k_cells<OBJ, SRC>, dim3(s.cluster, q.B), s.threads, s.smem, s.cluster, src, P);
    if (ev) for (int k = 1; k < 4; ++k) cudaEventRecord(ev[k], st);
    if (q.cells == 2) return;                                     // the caller looks at the flags itself
    SweepParams sp;
    sp.ts = q.ts; sp.meta = q.meta; sp.seg = q.seg;
    sp.n = q.n; sp.R = q.R; sp.B = q.B; sp.nseg = p.nseg; sp.nres = q.nres; sp.G = p.G_rest; sp.cap = p.cap;
    sp.flags = q.flags; sp.target = p.target_rest; sp.filter = 1;
    sp.need = nullptr;
    sp.max_rounds = q.max_rounds;
    FilterBufs f = fb;
    f.tailcap = 0x7fffffff;                                       // what the route finished is finished: finalize leaves it alone
    const long long items = std::max<long long>((long long)p.nseg * q.B, ((long long)q.n * q.B + CELL_REST_THREADS - 1) / CELL_REST_THREADS);
    launch(k_cell_rest<OBJ, SRC>, dim3((unsigned)std::max<long long>(1, std::min<long long>(q.num_sms, items))), CELL_REST_THREADS, p.smem, 1, src, sp, P, f);
    if (ev) cudaEventRecord(ev[4], st);
}

void enqueue_cells(const Pipeline &q, const FilterBufs &fb, const LaunchPlan &p, cudaStream_t st, cudaEvent_t *ev, const MatBatch &src) {
    if (q.objective == ZL_OBJ_RANGE) enqueue_cells_t<ZL_OBJ_RANGE>(q, fb, p, st, ev, src); else enqueue_cells_t<ZL_OBJ_SUM>(q, fb, p, st, ev, src);
}
void enqueue_cells(const Pipeline &q, const FilterBufs &fb, const LaunchPlan &p, cudaStream_t st, cudaEvent_t *ev, const AriBatch &src) {
    if (q.objective == ZL_OBJ_RANGE) enqueue_cells_t<ZL_OBJ_RANGE>(q, fb, p, st, ev, src); else enqueue_cells_t<ZL_OBJ_SUM>(q, fb, p, st, ev, src);
}

template <int OBJ, class SRC>
static cudaError_t cell_limits_t() {
    const int big = 200 * 1024;
    cudaError_t e = cudaFuncSetAttribute(k_cells<OBJ, SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cells<OBJ, SRC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cell_rest<OBJ, SRC>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    return e;
}

cudaError_t cell_limits() {
    cudaError_t e = cell_limits_t<ZL_OBJ_RANGE, MatBatch>();
    if (e == cudaSuccess) e = cell_limits_t<ZL_OBJ_RANGE, AriBatch>();
    if (e == cudaSuccess) e = cell_limits_t<ZL_OBJ_SUM, MatBatch>();
    if (e == cudaSuccess) e = cell_limits_t<ZL_OBJ_SUM, AriBatch>();
    return e;
}

}  // namespace zl
