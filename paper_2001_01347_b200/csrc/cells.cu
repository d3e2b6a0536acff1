// The cell route, both objectives, stored and predicted rows: no timestamp is sorted until it is known to matter, and of
// most rows only a few are read at all.
//
// The part of an instance's timeline that can hold the answer is cut into cells of a power of two of time units.  The
// search is branch and bound over the cells:
//   RANGE  The best Z whose minimum is at time t has max(Z) = G(t) = max over the rows of their first element at or after t,
//          so d = G(T) - T, and every candidate of a cell has d >= G(start) - end.  G is set by the rows with long
//          iterations: the slowest fifth to half of the rows ("guards": an eighth of the timestamps or so) give a lower bound of G
//          at every cell's start - a maximum per cell, then a prefix maximum; gaps much shorter than the smallest d that is to
//          be expected are passed over.  The cells with the smallest bounds are evaluated exactly (every row is asked for
//          its elements in them: eight elements where the row's ends suggest); the smallest d discards nearly all other cells,
//          and the ones it does not are evaluated the same way, runs of neighbours together, most promising first.  Where the
//          guards leave too many, the other rows are looked through for gaps longer than d: only those can discard a further cell.
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
// What bounds it: a call of one instance, the chain of some dozen dependent steps (0.5 to 2 us each); many instances, the
// instructions and latencies of looking through rows (2000 cycles for 32 pieces of eight elements with 20 warps an SM, n=1024,
// R=1024, B=64 16 of 37 us in the kernel), not what it moves (2.8 TB/s there).
//
// Times in this file are us a call of one seed's inputs that stay the same from call to call, unless said otherwise: they compare two ways of
// doing something.  With inputs that change a call takes longer (n=1024, R=1024, B=64 51 instead of 44 to 46, n=128, R=256, B=1024 43 instead of 37
// to 40), since nothing of the rows is in the L2.
//
// Every CTA of a cluster passes the same cluster barriers: whatever a loop or a branch around one depends on is the same
// value in the whole cluster (never the CTA's own number of rows or cells).
#include <cmath>
#include <cooperative_groups.h>

#include "zl_guard.cuh"
#include "zl_sweep.cuh"
#include "zl_host.h"

namespace cg = cooperative_groups;

namespace zl {

constexpr uint32_t INF32 = 0xffffffffu;
constexpr int CELL_ALIVE = 128;           // most cells of an instance that the bounds may leave
constexpr int CELL_BATCH = 16;            // most cells that the rows are asked for at once
constexpr int CELL_PAIRS = 256;           // answers that a batch of cells should give, from what the last ones gave
constexpr int CELL_CLUSTER = 16;          // most CTAs of a cluster
// The forms of the kernel.  ONE: an instance has one CTA, and what only clusters need falls away; THREADS: most threads of an SM, and so the
// registers of a thread; ROWS: rows that are looked through at a time, NODES: most elements in the cells that the rows are asked for at once.
// With 96 registers (640 threads) and with 72 nothing is spilled, with 80 20 bytes, with 64 48 bytes; a cluster's kernel with 72 or 64
// spills inside the loops, and what is spilled has often left the L1 cache, past which the rows stream, by the time it is wanted back (n=1024, R=1024,
// B=64 55 and 74 us, 44 with 96).  CTAs get registers for four warps at a time, so that 96 are good for five small CTAs an SM, 72 for seven: a thousand
// instances are one turn instead of 1.4 (n=128, R=256, B=1024 53 us with 96, 40 with 72; n=181, R=18, B=1795 60 / 54; predicted n=131, R=41,
// B=1760 44 / 37).  Three CTAs of 256 threads fit with 80 (n=350, R=157, B=373 53 us with 96 and 128 threads, 44 with 80), four with 64 (n=400, R=100,
// B=480 48 us with 96 and 128 threads, 43 with 64; n=22, R=537, B=565 54 / 49; but instances of 128 threads' work: n=30, R=60, B=580 28 / 31).
// With lists half as long (ROWS, NODES) there is room for 1400 cells more where seven CTAs share an SM.
// SUM, 128 threads of 96 registers / 256 of 80, three an SM (new inputs every call): n=256, R=256, B=300 282 / 194 us, n=300, R=300, B=330 167 / 127, n=128, R=128,
// B=400 59 / 48, n=64, R=30, B=440 24.2 / 23.2; of 64, four an SM: n=200, R=200, B=500 104 / 91, n=400, R=100, B=480 136 / 122, n=256, R=100, B=512 107 / 99;
// but instances of up to 64 timestamps a thread n=100, R=60, B=560 41.1 / 41.5, n=128, R=40, B=590 37.2 / 38.3.  (All with as many cells.)
template <bool ONE_, int THREADS_, int ROWS_, int NODES_>
struct CellForm { static constexpr bool ONE = ONE_; static constexpr int THREADS = THREADS_, ROWS = ROWS_, NODES = NODES_, CTAS = ONE_ ? 1 : CELL_CLUSTER; };
typedef CellForm<false, 640, 1024, 1024> CellCluster;
typedef CellForm<true, 640, 1024, 1024> CellAlone;        // up to two CTAs an SM, and SUM five and more
typedef CellForm<true, 768, 1024, 1024> CellThreeSum;     // SUM: three an SM,
typedef CellForm<true, 1024, 1024, 1024> CellFourSum;     // four
typedef CellForm<true, 768, 512, 512> CellThree;          // RANGE: three an SM,
typedef CellForm<true, 1024, 512, 512> CellFour;          // four, or eight,
typedef CellForm<true, 640, 512, 512> CellFive;           // four of 128 threads, or five,
typedef CellForm<true, 896, 512, 512> CellSeven;          // six or seven (or eight)
constexpr int CELL_FIRST = 4;             // most runs of cells that a round asks for at first
// Cells next to one another are asked for as one: the eight elements that a row is looked at for hold what it has in several cells as well.
// RUN: most cells of a run (a power of two); two cells of the list belong to one if there are at most RUN / 2 others between them.
template <int OBJ> constexpr uint32_t CELL_RUN = OBJ == ZL_OBJ_SUM ? 32 : 8;
constexpr long long CELL_ASK = 4;         // asking a row for a cell costs about as much as looking through this many of its elements, all cells of a
                                          // batch at once (n=1024, R=1024, B=64, mean of ten seeds 69 us with 16 and half the batch, 63 with 4)
constexpr int CELL_ROUNDS = 4;            // rounds after the first in which more cells may be left than there is room for (regular rows need one or two, SUM
                                          // up to four; with 48, rows of equal periods, n=64, R=128, took 0.5 ms before they were given up)
constexpr int CELL_HOPELESS = 2 * CELL_ALIVE;    // ... and so many are never worth a further round
// Runs of cells evaluated, eight for every round and one to sixteen answers (SUM 64), beyond which the handle's next calls leave the route:
// regular rows need up to 50 (RANGE; predicted rows of a common kind, n=20, R=185, B=1356) and 87 (SUM); where many cells tie the other routes are the
// faster ones (RANGE, times rounded to half a mean iteration, n=93, R=211, B=64 494 us / 99).
constexpr int CELL_ASKED_RANGE = 72, CELL_ASKED_SUM = 112;
constexpr int CELL_IDLE = 32;             // elements of a row in one cell that cannot matter, from which on the row is taken to stand still (one timestamp
                                          // everywhere, n=1024, R=1024, B=8 511 us / 58 on the filter route: one thread goes through them)
constexpr float CELL_OFF = 64.f;          // RANGE: elements by which a row's middle is off its estimate, root mean square, from which on the rows are far from
                                          // arithmetic: what the estimate misses is read by one thread, eight elements after the other (gaps with a power-law
                                          // tail, n=1024, R=1024, B=8 305 us / 60 on the filter route, bursts of iterations 301 / 70; but iterations that grow
                                          // fivefold, R=256 and 43 off, n=128, B=256 65 / 284)
constexpr int CELL_FEW = 8;               // so many cells are asked for in any case
constexpr int CELL_SLACK = 4;             // elements by which a row may be off its estimate before it is read on, at least
constexpr int EXPECTED_BINS = 2;          // RANGE: bins below the d to be expected from which on gaps are passed over (n=1024, R=1024, B=64 44.5 us, 46.2 when none
                                          // are, 43.8 with 0, but then n=1000, R=150, B=1 29 instead of 21: more cells are left)
constexpr int GUARD_BINS = 64;            // rows by their span, eight bins to a factor of two below the longest
constexpr float GUARD_IRREGULAR = 32.f;   // bins by which more rows are looked through, to a unit of their gaps' relative deviation above 0.1
constexpr float RANGE_CELLS = 100.f;      // RANGE: cells to the longest mean iteration
constexpr float SUM_WIDTH = 0.12f;        // SUM: n cell widths against the spread of the wait over time (see k_cells)

// ------------------------------------------------------------------------------ rows
// Relative times of an instance's rows, 32 bits: elements before the first are at time 0 (before everything), those behind
// the last infinite.  in(): one element known to exist.  load(): elements i .. i + 7 as they are stored, with i as given by
// align() (a 32-byte boundary of memory: two 32-byte loads), which rel() makes times of, and trim() sees to what lies
// outside the row.  load() has no branch - one whose sides meet again in the same registers makes the loads in it wait for
// each other -: pieces that the matrix does not have the memory for, at its very ends, are !whole() and hold something else.
template <class SRC> struct RowReader;
template <> struct RowReader<MatBatch> {
    const int64_t *inst; int R; uint32_t tminlo; int first, last;     // the piece that starts at element i + row * R exists from `first` to `last`
    __device__ __forceinline__ RowReader(const MatBatch &s, int b, int B, int n, int R_, int64_t tmin)
        : inst(s.ts + (size_t)b * n * R_), R(R_), tminlo((uint32_t)(uint64_t)tmin - 1u) {
        const int off = (int)(((uintptr_t)inst >> 3) & 3u);           // elements from the boundary before the instance to its first
        first = b > 0 ? -off : off ? 4 - off : 0;
        last = (int)min((long long)(B - b) * n * R_ - 8, 0x7ffffff0ll);
        last -= (last + off) & 3;                                     // (a matrix of fewer than eight elements: last < first)
    }
    __device__ __forceinline__ uint32_t in(int row, int i) const { return (uint32_t)(uint64_t)ldg64(inst + (size_t)row * R + i) - tminlo; }
    __device__ __forceinline__ uint32_t rel(uint64_t x) const { return (uint32_t)x - tminlo; }
    __device__ __forceinline__ bool whole(int row, int i) const { return row * R + i >= first && row * R + i <= last; }      // n * R is below 2^31
    __device__ __forceinline__ void load(int row, int i, uint64_t (&v)[8]) const {
        if (last < first) return;
        const int64_t *p = inst + min(max(row * R + i, first), last);
        asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
        asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[4]), "=l"(v[5]), "=l"(v[6]), "=l"(v[7]) : "l"(p + 4));
    }
    __device__ __forceinline__ int align(int row, int i) const { return i - (int)(((uintptr_t)(inst + (size_t)row * R + i) >> 3) & 3u); }
    __device__ __forceinline__ void prefetch(int row, int i) const {
        if (last < first) return;
        const int64_t *p = inst + min(max(row * R + i, first), last);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 4));
    }
};
template <> struct RowReader<AriBatch> {
    const int64_t *last, *iv; int R; uint32_t tminlo;
    __device__ __forceinline__ RowReader(const AriBatch &s, int b, int, int n, int R_, int64_t tmin)
        : last(s.last + (size_t)b * n), iv(s.iv + (size_t)b * n), R(R_), tminlo((uint32_t)(uint64_t)tmin - 1u) {}
    __device__ __forceinline__ uint32_t in(int row, int i) const {
        return (uint32_t)(uint64_t)ldg64(last + row) - tminlo + (uint32_t)(i + 1) * (uint32_t)(uint64_t)ldg64(iv + row);
    }
    __device__ __forceinline__ uint32_t rel(uint64_t x) const { return (uint32_t)x; }
    __device__ __forceinline__ void load(int row, int i, uint64_t (&v)[8]) const {
        const uint32_t d = (uint32_t)(uint64_t)ldg64(iv + row);
        uint32_t t = in(row, i);
#pragma unroll
        for (int k = 0; k < 8; ++k, t += d) v[k] = t;
    }
    __device__ __forceinline__ bool whole(int, int) const { return true; }
    __device__ __forceinline__ int align(int, int i) const { return i; }
    __device__ __forceinline__ void prefetch(int, int) const {}
};
template <class RD>
__device__ __forceinline__ uint32_t element(const RD &rd, int row, int i) { return i < 0 ? 0u : i < rd.R ? rd.in(row, i) : INF32; }
// Element i - 1 and the eight from i on, whatever is there.
template <class RD>
__device__ __forceinline__ void nine(const RD &rd, int row, int i, uint32_t (&T)[9]) {
#pragma unroll
    for (int k = 0; k < 9; ++k) T[k] = element(rd, row, i - 1 + k);
}
// T[1] to T[8] of eight loaded elements, i the first of them.
template <class RD>
__device__ __forceinline__ void trim(const RD &rd, int i, const uint64_t (&v)[8], uint32_t (&T)[9]) {
#pragma unroll
    for (int k = 0; k < 8; ++k) T[k + 1] = rd.rel(v[k]);
    if (i < 0 || i + 8 > rd.R) {
#pragma unroll
        for (int k = 0; k < 8; ++k) { if (i + k < 0) T[k + 1] = 0u; if (i + k >= rd.R) T[k + 1] = INF32; }
    }
}

// ------------------------------------------------------------------------------ reductions of a warp
// 64 bits as two 32-bit reductions of the hardware (five shuffle steps of two registers take several times as long).
__device__ __forceinline__ uint64_t warp_min64(uint64_t v) {
    const uint32_t h = __reduce_min_sync(FULL, (uint32_t)(v >> 32));
    return (uint64_t)h << 32 | __reduce_min_sync(FULL, (uint32_t)(v >> 32) == h ? (uint32_t)v : INF32);
}
__device__ __forceinline__ uint64_t warp_max64(uint64_t v) {
    const uint32_t h = __reduce_max_sync(FULL, (uint32_t)(v >> 32));
    return (uint64_t)h << 32 | __reduce_max_sync(FULL, (uint32_t)(v >> 32) == h ? (uint32_t)v : 0u);
}
// (pieces of 26, 26 and 12 bits: a sum of 32 of them fits)
__device__ __forceinline__ uint64_t warp_sum64(uint64_t v) {
    const uint32_t m = (1u << 26) - 1u;
    return (uint64_t)__reduce_add_sync(FULL, (uint32_t)v & m) + ((uint64_t)__reduce_add_sync(FULL, (uint32_t)(v >> 26) & m) << 26) +
           ((uint64_t)__reduce_add_sync(FULL, (uint32_t)(v >> 52)) << 52);
}
__device__ __forceinline__ float warp_sum(float x) {              // the same value in every lane
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(FULL, x, d);
    return x;
}

// ------------------------------------------------------------------------------ looking through rows
// The rows that have elements in the time range [a, b) of interest, and the pieces of eight elements that each of them needs:
// a row's pieces are sb + 8 q with q from excl up to the next row's.  In shared memory, a batch of rows at a time.
template <int ROWS_>
struct RowList {
    static constexpr int ROWS = ROWS_;
    uint32_t excl[ROWS];
    int sb[ROWS];
    unsigned short row[ROWS];
};

// A row (a lane; `have`: it counts) goes to the list.  Which pieces it needs is estimated from its ends, `slack` elements more on
// either side: rows are close to arithmetic.  fill: rows and pieces so far, in one word of 32 bits where pieces are sure to fit
// into 20 of them (64-bit atomics on shared memory are loops).  The warp's lanes call together.
struct ListFill { uint32_t packed; unsigned long long wide; };
constexpr int LIST_BITS = 20;
__device__ __forceinline__ bool list_packed(int rows, int R) { return (long long)rows * (R / 8 + 3) < (1 << LIST_BITS); }
template <class LIST, class RD>
__device__ __forceinline__ void list_rows(LIST &L, ListFill &fill, bool packed, const RD &rd, int R, int row, bool have, uint32_t e0, uint32_t eR,
                                          uint32_t a, uint32_t b, int slack) {
    const int lane = threadIdx.x & 31;
    const unsigned who = __ballot_sync(FULL, have);
    if (!who) return;
    int s0 = 0;
    uint32_t np = 0;
    if (have) {
        const float f = eR > e0 ? (float)(R - 1) / (float)(eR - e0) : 0.f;
        if (a > e0) s0 = max(0, min((int)((float)(a - e0) * f) - slack, R - 1));
        s0 = rd.align(row, s0);
        const int last = b > eR ? R : min((int)((float)(b - e0) * f) + 1 + slack, R);
        np = (uint32_t)max(1, (last - s0 + 8) >> 3);
    }
    uint32_t incl = np;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, incl, d); if (lane >= d) incl += y; }
    uint32_t rows = 0, q = 0;
    if (lane == 31) {
        if (packed) {
            const uint32_t at = atomicAdd(&fill.packed, (uint32_t)__popc(who) << LIST_BITS | incl);
            rows = at >> LIST_BITS; q = at & ((1u << LIST_BITS) - 1u);
        } else {
            const unsigned long long at = atomicAdd(&fill.wide, (unsigned long long)__popc(who) << 40 | incl);
            rows = (uint32_t)(at >> 40); q = (uint32_t)at;
        }
    }
    rows = __shfl_sync(FULL, rows, 31); q = __shfl_sync(FULL, q, 31);
    if (have) {
        const int pos = (int)rows + __popc(who & ((1u << lane) - 1u));
        q += incl - np;
        L.excl[pos] = q; L.sb[pos] = (int)((uint32_t)s0 - 8u * q); L.row[pos] = (unsigned short)row;
    }
}

// The CTA looks through the listed rows: the pieces are dealt out evenly to its warps, each a run of them, a piece a lane.
// (Rows dealt out instead, 32 to a warp, leave the warps with the most guards twice as long at it as the others: n=1024, R=1024,
// B=64 14 to 25 us for this pass.  A run of pieces a thread scatters the loads: n=4096, R=4096, B=8 327 us a call instead of 161.)  While one
// is worked on, the lane's next is on its way to the L2.  Where the estimate of a row's pieces falls short on either side its
// first or last piece leaves a bit, and all such rows are read on by the whole CTA at the end (one access after the other by
// the lane itself, with its warp waiting, takes half as long again where single gaps are long).  act(T) gets nine consecutive
// times, eight pairs of neighbours: every pair with one of its elements in the range, and the pair that straddles a, comes
// exactly once; others may come.
template <class LIST, class RD, class ACT>
__device__ __forceinline__ void stream_list(const LIST &L, uint32_t (*more)[LIST::ROWS / 32], int rows, uint32_t pieces, const RD &rd, int R, uint32_t a, uint32_t b, ACT act) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t share = (pieces + nw - 1) / nw, p0 = min(share * warp, pieces), p1 = min(p0 + share, pieces);
    if (p0 < p1) {
        // the row that piece p0 belongs to: the last one that starts at or before it, two steps of 32
        int j0;
        {
            const int per = (rows + 31) / 32;
            const unsigned m = __ballot_sync(FULL, lane * per < rows && L.excl[min(lane * per, rows - 1)] <= p0);
            j0 = (__popc(m) - 1) * per;
            const unsigned k = __ballot_sync(FULL, lane < per && j0 + lane < rows && L.excl[min(j0 + lane, rows - 1)] <= p0);
            j0 += __popc(k) - 1;                                      // LIST::ROWS <= 32 * 32
        }
        // piece q + lane: its entry of the list, its first element, whether it is its row's first (1) or last (2) one
        auto assign = [&](uint32_t q, int &entry, int &s, unsigned &edge) {
            const int j = j0 + lane;
            const uint32_t h = (j < rows ? L.excl[j] : pieces) - q;   // where the lane's entry starts; entry j0 at or before q
            const unsigned heads = __reduce_or_sync(FULL, h < 32u ? 1u << h : 0u);      // (bit 0: entry j0 starts with piece q)
            const int k = __popc((heads & ~1u) & (FULL >> (31 - lane))), behind = j0 + __popc(heads & ~1u) + 1;
            const bool next = (behind < rows ? L.excl[behind] : pieces) == q + 32u;     // a row, or the end, right behind these 32
            entry = min(j0 + k, rows - 1);
            s = (int)((uint32_t)L.sb[entry] + 8u * (q + lane));
            edge = ((heads >> lane) & 1u) | ((lane < 31 ? (heads >> (lane + 1)) & 1u : next ? 1u : 0u) << 1);
            j0 = behind - (next ? 0 : 1);
        };
        int entry, s;
        unsigned edge;
        assign(p0, entry, s, edge);
        // (lane 0) the element before the first of these pieces.  The other lanes may have no piece, and their s lies behind the row.
        uint32_t carry = 0;
        if (lane == 0) carry = rd.in(L.row[entry], max(s - 1, 0));
#pragma unroll 1
        for (uint32_t q = p0; q < p1; q += 32u) {
            const uint32_t x = q + lane;
            const bool mine = x < p1;
            const int row = L.row[entry];
            uint64_t v[8];
            if (mine) rd.load(row, s, v);
            int nentry = 0, ns = 0;
            unsigned nedge = 0;
            if (q + 32u < p1) {                                       // the next piece on its way to the L2 while this one is worked on
                assign(q + 32u, nentry, ns, nedge);
                if (x + 32u < p1) rd.prefetch(L.row[nentry], ns);
            }
            uint32_t T[9];
            trim(rd, s, v, T);
            if (mine && !rd.whole(row, s)) nine(rd, row, s, T);       // (seldom)
            const uint32_t up = __shfl_up_sync(FULL, T[8], 1);
            T[0] = (edge & 1u) ? (s > 0 ? T[1] : 0u) : lane == 0 ? carry : up;      // (a row's first piece starts with no gap: see below)
            carry = __shfl_sync(FULL, T[8], 31);
            if (mine) {
                act(T);
                if ((edge & 1u) && s > 0 && T[1] >= a) atomicOr(&more[0][entry >> 5], 1u << (entry & 31));
                if ((edge & 2u) && s + 8 <= R && T[8] < b) atomicOr(&more[1][entry >> 5], 1u << (entry & 31));
            }
            entry = nentry; s = ns; edge = nedge;
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int i = threadIdx.x; i < 2 * LIST::ROWS; i += blockDim.x) {
        const int right = i >= LIST::ROWS ? 1 : 0, j = i & (LIST::ROWS - 1);
        if (j < rows && (more[right][j >> 5] >> (j & 31) & 1u)) {
            const int row = L.row[j];
            int s = (int)((uint32_t)L.sb[j] + 8u * (right ? (j + 1 < rows ? L.excl[j + 1] : pieces) - 1u : L.excl[j]));
            if (!right) ++s;                                      // to the left the pair of the piece's first element and the one before it comes along
            bool on = true;
#pragma unroll 1
            while (on) {
                uint32_t U[9];
                s += right ? 8 : -8;
                nine(rd, row, s, U);
                act(U);
                on = right ? s + 8 <= R && U[8] < b : s > 0 && U[0] >= a;
            }
        }
    }
}

// Where the eight elements that are looked at first for time t start: t's place by the row's ends, a little before it.
template <class RD>
__device__ __forceinline__ int window_at(const RD &rd, int row, int R, uint32_t t, uint32_t e0, float inv) {
    return rd.align(row, min(max((t > e0 ? (int)min((float)(t - e0) * inv, (float)R) : 0) - 2, 0), R - 1));
}
__device__ __forceinline__ float per_time(int R, uint32_t e0, uint32_t eR) { return eR > e0 ? (float)(R - 1) / (float)(eR - e0) : 0.f; }
// They start at s and do not hold the first element at or after a, or not the one before it, or not all up to what is asked for: where the
// next eight start, by how far off these are.
template <class RD>
__device__ __forceinline__ int window_next(const RD &rd, int row, int R, int s, uint32_t T1, uint32_t T8, uint32_t a, float inv) {
    const int off = (int)min((float)(T1 >= a ? T1 - a : T8 < a ? a - T8 : 0u) * inv, (float)R);
    return rd.align(row, min(max(T1 >= a ? s - 3 - off : T8 < a ? s + 5 + off : s + 4, 0), R - 1));
}

// Index of a row's first element at or after time t, by one thread: eight elements around the place that the row's ends suggest, then
// where the mean interval puts t from the nearest of those; then bisection.
template <class RD>
__device__ __noinline__ int first_at_or_after(const RD rd, int row, int R, uint32_t t, uint32_t e0, uint32_t eR) {
    if (t <= e0) return 0;
    if (t > eR) return R;
    int lo = 0, hi = R - 1;                                       // element lo is before t, element hi is not (e0 < t <= eR)
    const float inv = per_time(R, e0, eR);
    int s = window_at(rd, row, R, t, e0, inv);
#pragma unroll 1
    for (int it = 0; it < 4 && rd.whole(row, s); ++it) {
        uint64_t v[8];
        uint32_t T[9];
        rd.load(row, s, v);
        trim(rd, s, v, T);
        int c = 0;
#pragma unroll
        for (int k = 1; k < 9; ++k) c += T[k] < t ? 1 : 0;        // sorted: the first c of them
        if (c < 8 && (c > 0 || s <= lo + 1)) return s + c;
        if (c == 0) hi = min(hi, s); else lo = max(lo, s + 7);
        s = rd.align(row, min(max(window_next(rd, row, R, s, T[1], T[8], t, inv), lo), hi));
    }
#pragma unroll 1
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (rd.in(row, mid) < t) lo = mid; else hi = mid;
    }
    return hi;
}

// Whether one of `rows` consecutive rows decreases somewhere: their elements one after the other, whatever rows they belong
// to, 512 a warp and step with four 32-byte loads a lane under way.  (A warp a row: the next row's loads wait for this one's, n=93,
// R=211 5.6 us; eight 8-byte loads a lane: n=1111, R=1072, B=44 134 us.)
static __device__ bool rows_unsorted(const int64_t *ts, int rows, int R) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long N = (long long)rows * R;                      // (n * R is below 2^31)
    bool bad = false;
    // up to the first 32-byte boundary and behind the last whole 512 (or, rows shorter than eight, all): an element a thread
    const int head = R < 8 ? (int)N : (int)min((long long)((4u - (unsigned)((uintptr_t)ts >> 3)) & 3u), N);
    const int steps = (int)((N - head) >> 9);
    for (long long f = threadIdx.x; f < N; f += blockDim.x) {
        const long long end = head + 512ll * steps;
        if (f >= head && f < end) {                               // (the steps' own)
            f += (end - f) / blockDim.x * blockDim.x;
            if (f < end) continue;
            if (f >= N) break;
        }
        bad |= (uint32_t)f % (uint32_t)R != 0u && ldg64(ts + f) < ldg64(ts + f - 1);
    }
#pragma unroll 1
    for (int k = warp; k < steps; k += nw) {
        const int f0 = head + 512 * k;
        int64_t v[2][8], before = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t *p = ts + f0 + 256 * u + 8 * lane;
            asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[u][0]), "=l"(v[u][1]), "=l"(v[u][2]), "=l"(v[u][3]) : "l"(p));
            asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(v[u][4]), "=l"(v[u][5]), "=l"(v[u][6]), "=l"(v[u][7]) : "l"(p + 4));
        }
        if (lane == 0 && f0 > 0) before = ldg64(ts + f0 - 1);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            int64_t up = (int64_t)shfl_up((uint64_t)v[u][7], 1);
            if (lane == 0) up = before;
            before = (int64_t)shfl_idx((uint64_t)v[u][7], 31);
            // which of the eight starts a row, and so follows nothing
            const int c = (int)((uint32_t)(f0 + 256 * u + 8 * lane) % (uint32_t)R), first = c == 0 ? 0 : R - c;
            bad |= first != 0 && v[u][0] < up;
#pragma unroll
            for (int j = 1; j < 8; ++j) bad |= first != j && v[u][j] < v[u][j - 1];
        }
    }
    return bad;
}

// ------------------------------------------------------------------------------ checked rows
// Stored rows, every load checked against the instance (single elements) or the matrix (pieces of eight): a bad index is recorded and the
// load skipped.  For handles with ZL_FLAG_DEBUG_CHECKS that are told to take the route.
struct MatChecked {
    const int64_t *ts; uint32_t *record;
    typedef MatRows Rows;
    __device__ __forceinline__ MatRows inst(int b, int n, int R) const { return MatRows{ts + (size_t)b * n * R, R}; }
};
template <> struct RowReader<MatChecked> : RowReader<MatBatch> {
    Guard<true> guard; long long before, own, all;                // elements of the matrix before the instance, of the instance, of the matrix
    __device__ __forceinline__ RowReader(const MatChecked &s, int b, int B, int n, int R_, int64_t tmin)
        : RowReader<MatBatch>(MatBatch{s.ts}, b, B, n, R_, tmin), guard{s.record, blockIdx.y * gridDim.x + blockIdx.x},
          before((long long)b * n * R_), own((long long)n * R_), all((long long)B * n * R_) {}
    __device__ __forceinline__ uint32_t in(int row, int i) const {
        return guard.ok((uint64_t)((long long)row * R + i), (uint64_t)own, ACC_ROW) ? RowReader<MatBatch>::in(row, i) : 0u;
    }
    __device__ __forceinline__ void load(int row, int i, uint64_t (&v)[8]) const {
        const long long at = before + min(max(row * R + i, first), last);
        if (last >= first && guard.ok((uint64_t)at, (uint64_t)max(all - 7, 0ll), ACC_ROW_PIECE) &&
            guard.ok((uintptr_t)(inst + (at - before)) & 31u, 1, ACC_ROW_ALIGN)) {
            RowReader<MatBatch>::load(row, i, v);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = 0;
        }
    }
};
__host__ __device__ inline MatBatch plain_rows(const MatChecked &s) { return MatBatch{s.ts}; }
template <class SRC> __host__ __device__ inline SRC plain_rows(const SRC &s) { return s; }

// ------------------------------------------------------------------------------ the search
struct CellParams {
    int n, R, B;
    int cap;                         // cells a CTA has room for (a multiple of 128)
    int rpc;                         // rows of a CTA when rows are asked
    int check_sorted;                // every row is read once to see that it does not decrease
    int near;                        // the rows are in this GPU's memory (across the bus every timestamp read in vain costs more than reading on)
    InstMeta *meta;
    uint32_t epoch;                  // number of the call: a word of `flags` is raised when it holds this
    uint32_t *flags;                 // [1] some instance needs the segment sweep, [2] some instance's outputs are missing,
                                     // [3] the calls to come should rather not take this route, [4], [5] grid_barrier
    int32_t *idx; int64_t *barrier; int64_t *wait; int32_t *status;
};

// What the rows answer when they are asked for cells.  A cluster has three of them: what the own rows answered, and what arrived from
// every CTA (its share of the room each), twice, used in turn: the next answers may arrive while these are worked on.
template <int NODES>
struct Answers {
    uint64_t node[NODES];                         // the elements in the cells: time << 32 | RANGE the row's next element, SUM the element less the row's previous one
    unsigned char slot[NODES];                    // ... which of the cells
};

template <int OBJ, class FORM>
struct CellShared {
    typedef typename std::conditional<OBJ == ZL_OBJ_RANGE, uint32_t, unsigned long long>::type Sum;      // RANGE: a time, SUM: a sum of times
    // from every CTA of the cluster (each array is written by the others before one cluster barrier and read after it, so no
    // two exchanges share one): minima and maxima of its rows' ends; whether one of its rows decreases; SUM its rows' wait at
    // the sample time; the key of its best cell, and G or S at its start
    unsigned long long ex[4][FORM::CTAS];
    float exi[FORM::CTAS];                      // RANGE: how irregular its rows are (sum over a few of them, see k_cells)
    unsigned long long exc[FORM::CTAS], exs[FORM::CTAS], exv[FORM::CTAS], exb[FORM::CTAS];
    unsigned long long red[4][32], keys[32], kbases[32];
    // of Answers: how many from every CTA; RANGE latest and earliest of the rows' first elements at or after the cell's start
    struct { uint32_t gmax[CELL_BATCH], gmin[CELL_BATCH]; uint32_t count[FORM::CTAS]; } heard[FORM::ONE ? 1 : 2];
    uint32_t gmax[CELL_BATCH], gmin[CELL_BATCH];  // ... of the own rows'
    unsigned int nnodes;
    ListFill fill;
    unsigned long long acc, total;
    uint32_t hist[GUARD_BINS];
    unsigned long long later;                     // RANGE: about how many timestamps of the other rows lie in the range
    // the cells to evaluate (in every CTA), and the order in which that is done
    uint32_t cell[CELL_ALIVE];
    union {
        struct {
            Sum base[CELL_ALIVE];                 // RANGE: a lower bound of G at the cell's start, SUM: S there
            Sum lb[CELL_ALIVE];                   // lower bound of the objective in the cell
        };
        uint32_t more[2][FORM::ROWS / 32];         // (while rows are looked through: which of them have to be read on, to the left, to the right)
    };
    unsigned short order[CELL_ALIVE];
    unsigned int ncells;
    // the ones that the rows are being asked for: first and last time, G or S as above
    uint32_t ca[CELL_BATCH], ce[CELL_BATCH];
    uint64_t cb[CELL_BATCH];
    uint2 asked_run[CELL_FIRST * (CELL_ROUNDS + 2)];      // first and last cell of the runs evaluated before the list was made
    // the list's runs, in the order of their first cells: first and last cell, G or S at the start, smallest lower bound
    uint2 run[CELL_ALIVE];
    Sum run_base[CELL_ALIVE];
    unsigned long long run_lb[CELL_ALIVE];        // (64 bits in any case: with 32 the compiler spills twenty registers where it has 72)
    uint32_t exf[FORM::CTAS];                   // (exchanged with exv, exb) first cell of the run around the most promising one
    int runs;
    uint64_t bestd[32]; uint32_t bestt[32];
    // what is the same in all threads and needed now and then: shared memory, not a register each (the compiler spills some sixty of
    // them otherwise, and what is spilled has often left the L1 cache by the time it is wanted back: n=1024, R=1024, B=64 72 us)
    int64_t tmin;
    uint64_t ub, bd;                              // SUM: a wait that is attained; the smallest objective so far and its time
    uint32_t bt, t0, lmin, tend, lo, hi, shift, c0, m, a, bnd, gap, took;
    float span, width;                            // RANGE: rows of at least this span are guards; what a cell may span
    int slack, firsts, around, ndone, asked, per_cell;
    unsigned int slow;                            // (in every CTA) rows far from arithmetic, or standing still
};

// A cell's last time; `limit` is where the timeline (or a CTA's slice of it) ends.  Formed from what is left of it behind the
// cell's start: start + width would pass 2^32 in the last cell of a timeline that ends just below.
__device__ __forceinline__ uint32_t cell_end(uint32_t start, uint32_t shift, uint32_t limit) {
    return start + min((1u << shift) - 1u, limit - 1u - start);
}

static __device__ __noinline__ bool was_asked(const uint2 *runs, int n, uint32_t c) {
    bool is = false;
#pragma unroll 1
    for (int k = 0; k < n; ++k) is |= runs[k].x <= c && c <= runs[k].y;
    return is;
}

// The same variable in CTA `rank` of the cluster.  (ONE: the instance has one CTA.)
template <bool ONE, class T> __device__ __forceinline__ T *map_shared_rank(T *x, int rank) {
    if constexpr (ONE) return x; else return cg::this_cluster().map_shared_rank(x, rank);
}

struct Best { uint64_t d; uint32_t t; };          // smallest objective and its time, the first of equal ones; the same in every thread of the cluster
__device__ __forceinline__ Best warp_best(uint64_t d, uint32_t t) {
    const uint64_t m = warp_min64(d);
    return Best{m, __reduce_min_sync(FULL, d == m ? t : INF32)};
}

// The exact minimum over the `ns` cells of sh.ca, sh.ce, sh.cb (in every CTA of the cluster the same): every CTA asks its rows
// and sends what they answer to all CTAs, and behind one cluster barrier every CTA (with a few dozen answers every
// warp, without a further barrier) evaluates all of it.  Every thread of the cluster calls.  Returns the number of answers: more than FORM::NODES,
// and there was no room for them.
//
// A (cell, row) pair a lane, a warp on one cell: eight elements around the place that the row's ends suggest are loaded, then,
// by how far off they were, eight others, until they hold the first element at or after the cell's start and all that
// follow in it.  (Searched for the first element, then asked for its successor and the next ones: three to five accesses one
// after the other, n=1024, R=1024, B=64 7 us, eight cells of SUM 17 us.)
template <int OBJ, class SRC, class FORM>
__device__ __forceinline__ int evaluate_cells(CellShared<OBJ, FORM> &sh, Answers<FORM::NODES> *answers, const uint2 *ends, const SRC &src, int B, int n, int R, int rpc, int turn, int ns) {
    cg::cluster_group cl = cg::this_cluster();
    constexpr bool ONE = FORM::ONE;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5, G = ONE ? 1 : gridDim.x;
    const int r0 = ONE ? 0 : min((int)blockIdx.x * rpc, n), nrows = ONE ? n : min(rpc, n - r0);
    const RowReader<SRC> rd(src, blockIdx.y, B, n, R, sh.tmin);
    typedef Answers<FORM::NODES> Ans;
    Ans *an = answers;
    auto put = [&](int k, uint32_t T, uint32_t pay) {
        const unsigned pos = atomicAdd(&sh.nnodes, 1u);
        if (pos < FORM::NODES) { an->node[pos] = (uint64_t)T << 32 | pay; an->slot[pos] = (unsigned char)k; }
    };
    const int chunks = (rpc + 31) >> 5, items = ns * chunks;
#pragma unroll 1
    for (int it = warp; it < items; it += nw) {
        const int k = it / chunks, p = 32 * (it - k * chunks) + lane, row = r0 + p;
        const uint32_t a = sh.ca[k], e = sh.ce[k];
        const uint64_t base = sh.cb[k];
        uint32_t first = 0, last = INF32;                         // RANGE: of the row, for the latest and the earliest
        if (p < nrows) {
            const uint2 en = ends[row];
            const float inv = per_time(R, en.x, en.y);
            int s = window_at(rd, row, R, a, en.x, inv);
            uint32_t T[9];
            bool open = true;
#pragma unroll 1
            for (int step = 0; step < 4 && open; ++step) {
                uint64_t v[8];
                rd.load(row, s, v);
                trim(rd, s, v, T);
                if (!rd.whole(row, s)) break;
                open = !((T[1] < a || s <= 0) && T[8] > e);
                if (open) s = window_next(rd, row, R, s, T[1], T[8], a, inv);
            }
            if (!open) {
                T[0] = 0;
                uint32_t f = T[8];
                unsigned in = 0;                                  // which of the eight are answers
#pragma unroll
                for (int j = 7; j > 0; --j) {
                    if (T[j] >= a) f = T[j];
                    // (RANGE: an element that does not raise the running maximum cannot matter)
                    if (T[j] - a <= e - a && (OBJ == ZL_OBJ_RANGE ? (uint64_t)T[j + 1] > base : T[j] != T[j - 1])) in |= 1u << j;
                }
                first = last = f;
#pragma unroll 1
                for (; in; in &= in - 1u) {
                    const int j = __ffs(in) - 1;
                    uint32_t x = 0, y = 0;                        // RANGE elements j and j + 1, SUM j and j - 1
#pragma unroll
                    for (int i = 1; i < 8; ++i) if (i == j) { x = T[i]; y = T[OBJ == ZL_OBJ_RANGE ? i + 1 : i - 1]; }
                    put(k, x, OBJ == ZL_OBJ_RANGE ? y : x - y);
                }
            } else {
                int i = first_at_or_after(rd, row, R, a, en.x, en.y);
                uint32_t X = element(rd, row, i), pv = OBJ == ZL_OBJ_SUM ? element(rd, row, i - 1) : 0u;
                first = last = X;
                int idle = 0;
#pragma unroll 1
                for (; i < R && X <= e; ++i) {
                    const uint32_t nx = element(rd, row, i + 1);
                    const uint32_t pay = OBJ == ZL_OBJ_RANGE ? nx : X - pv;
                    if (OBJ == ZL_OBJ_RANGE ? (uint64_t)nx > base : pay != 0u) put(k, X, pay);
                    else if (++idle == CELL_IDLE) sh.slow = 1;
                    pv = X; X = nx;
                }
            }
        }
        if (OBJ == ZL_OBJ_RANGE) {
            first = __reduce_max_sync(FULL, first);
            last = __reduce_min_sync(FULL, last);
            if (lane == 0) { atomicMax(&sh.gmax[k], first); atomicMin(&sh.gmin[k], last); }
        }
    }
    __syncthreads();
    int m = (int)sh.nnodes, mine_k = 0;
    uint64_t mine_x = 0;
    const uint32_t *gmax = sh.gmax, *gmin = sh.gmin;
    if (G > 1) {
        const int rank = blockIdx.x, room = FORM::NODES / G, sent = min(m, room);
        auto &heard = sh.heard[turn];
        Ans *in = answers + 1 + turn;
        gmax = heard.gmax; gmin = heard.gmin;
#pragma unroll 1
        for (int r = warp; r < G; r += nw) {                      // to CTA r
            Ans *to = map_shared_rank<ONE>(in, r);
            for (int i = lane; i < sent; i += 32) { to->node[rank * room + i] = an->node[i]; to->slot[rank * room + i] = an->slot[i]; }
            auto *h = map_shared_rank<ONE>(&heard, r);
            if (lane == 0) h->count[rank] = (uint32_t)m;
            if (OBJ == ZL_OBJ_RANGE && lane < ns) { atomicMax(&h->gmax[lane], sh.gmax[lane]); atomicMin(&h->gmin[lane], sh.gmin[lane]); }
        }
        cl.sync();
        const int c = lane < G ? (int)heard.count[min(lane, G - 1)] : 0;
        int incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const int y = __shfl_up_sync(FULL, incl, d); if (lane >= d) incl += y; }
        m = __shfl_sync(FULL, incl, 31);
        const bool over = __any_sync(FULL, c > room);            // more from one CTA than its share: they are fetched from where they were put
        if (m <= 32 && !over) {
            // a lane each: from which CTA, and which of its answers
            int at = lane;
#pragma unroll 1
            for (int r = 0; r + 1 < G; ++r) { const int p = __shfl_sync(FULL, incl, r); if (lane >= p) at = (r + 1) * room + lane - p; }
            if (lane < m) { mine_x = in->node[at]; mine_k = in->slot[at]; }
        } else if (m <= FORM::NODES) {
            Ans *to = over ? in : an;
#pragma unroll 1
            for (int r = warp; r < G; r += nw) {
                const int count = __shfl_sync(FULL, c, r), at = __shfl_sync(FULL, incl, r) - count;
                const Ans *from = over ? map_shared_rank<ONE>(an, r) : in;
                const int first = over ? 0 : r * room;
                for (int i = lane; i < count; i += 32) { to->node[at + i] = from->node[first + i]; to->slot[at + i] = from->slot[first + i]; }
            }
            if (over) cl.sync(); else __syncthreads();
            an = to;
        }
    } else if (lane < m && m <= 32) {
        mine_x = an->node[lane]; mine_k = an->slot[lane];
    }
    uint64_t d = sh.bd;
    uint32_t t = sh.bt;
    if (OBJ == ZL_OBJ_RANGE && m <= FORM::NODES && lane < ns && gmax[lane] != INF32 && gmin[lane] < sh.hi) {
        // the first element at or after the cell's start, wherever it is
        const uint64_t w = (uint64_t)(gmax[lane] - gmin[lane]);
        if (w < d || (w == d && gmin[lane] < t)) { d = w; t = gmin[lane]; }
    }
    // the exact objective of an answer: the sweep over its cell's answers up to it.  Up to 32 of them: a lane each, every warp for itself.
    const bool few = m <= 32;
    if (few) {
        const uint32_t T = (uint32_t)(mine_x >> 32), pay = (uint32_t)mine_x;
        uint64_t v = lane < m ? (OBJ == ZL_OBJ_RANGE ? (uint64_t)gmax[mine_k] : sh.cb[mine_k]) : 0ull;
        // (RANGE: what G has at the start already does not raise it)
        const bool counts = lane < m && (OBJ == ZL_OBJ_SUM || pay > v);
        unsigned left = __ballot_sync(FULL, counts);
#pragma unroll 2
        for (; left; left &= left - 1u) {
            const int j = __ffs(left) - 1, k = __shfl_sync(FULL, mine_k, j);
            const uint32_t o = __shfl_sync(FULL, T, j), y = __shfl_sync(FULL, pay, j);
            if (OBJ == ZL_OBJ_RANGE) { if (k == mine_k && o < T) v = max(v, (uint64_t)y); }      // max(Z): latest next of the earlier elements
            else if (k == mine_k && o <= T) v += y;                                              // S: every delta up to T
        }
        const uint64_t w = OBJ == ZL_OBJ_SUM ? (uint64_t)n * T - v : v >= INF32 ? ~0ull : v - T;
        if (counts && w != ~0ull && (w < d || (w == d && T < t))) { d = w; t = T; }
    } else if (m <= FORM::NODES) {
#pragma unroll 1
        for (int i = tid; i < m; i += nt) {
            const uint64_t x = an->node[i];
            const uint32_t T = (uint32_t)(x >> 32);
            const int k = an->slot[i];
            uint64_t v = OBJ == ZL_OBJ_RANGE ? (uint64_t)gmax[k] : sh.cb[k];
#pragma unroll 8
            for (int j = 0; j < m; ++j) {
                const uint64_t y = an->node[j];
                const uint32_t o = (uint32_t)(y >> 32), pay = (uint32_t)y;
                const bool same = an->slot[j] == k;
                if (OBJ == ZL_OBJ_RANGE) { if (same && o < T) v = max(v, (uint64_t)pay); }
                else if (same && o <= T) v += pay;
            }
            const uint64_t w = OBJ == ZL_OBJ_SUM ? (uint64_t)n * T - v : v >= INF32 ? ~0ull : v - T;
            if (w != ~0ull && (w < d || (w == d && T < t))) { d = w; t = T; }
        }
    }
    Best best = warp_best(d, t);
    if (!few && m <= FORM::NODES) {
        if (lane == 0) { sh.bestd[warp] = best.d; sh.bestt[warp] = best.t; }
        __syncthreads();
        best = warp_best(lane < nw ? sh.bestd[lane] : ~0ull, lane < nw ? sh.bestt[lane] : INF32);
    }
    __syncthreads();                                              // everybody has read the answers
    if (tid == 0) { sh.nnodes = 0; sh.bd = best.d; sh.bt = best.t; sh.per_cell = max(1, m / ns); sh.asked += m / (OBJ == ZL_OBJ_RANGE ? 16 : 64); }
    if (tid < CELL_BATCH) { const int u = ONE ? 0 : turn; sh.gmax[tid] = sh.heard[u].gmax[tid] = 0; sh.gmin[tid] = sh.heard[u].gmin[tid] = INF32; }
    __syncthreads();
    return m;
}

// The elements of the slice's rows into its cells: RANGE of the guards (stage 0) or of the other rows (stage 1), SUM of all rows.
template <int OBJ, class SRC, class FORM>
__device__ __forceinline__ void look_through(CellShared<OBJ, FORM> &sh, uint32_t *cell, Answers<FORM::NODES> *answers, const uint2 *ends, const SRC &src, int B, int n, int R, int stage) {
    const RowReader<SRC> rd(src, blockIdx.y, B, n, R, sh.tmin);
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const uint32_t a = sh.a, bnd = sh.bnd, shift = sh.shift, gap = sh.gap, m = sh.m, w = bnd - a;
    uint64_t carry = 0, total = 0;                        // SUM: the rows' last elements before a, and all deltas in the slice
    RowList<FORM::ROWS> &list = *reinterpret_cast<RowList<FORM::ROWS> *>(answers);
    const bool packed = list_packed(min(n, FORM::ROWS), R);
#pragma unroll 1
    for (int from = 0; from < n && m > 0; from += FORM::ROWS) {
        if (from > 0) __syncthreads();
        if (tid < FORM::ROWS / 32) sh.more[0][tid] = sh.more[1][tid] = 0;
#pragma unroll 1
        for (int g = warp; 32 * g < min(FORM::ROWS, n - from); g += nw) {
            const int row = from + 32 * g + lane;
            uint2 e = make_uint2(0u, 0u);
            bool have = row < n;
            if (have) {
                e = ends[row];
                if (OBJ == ZL_OBJ_RANGE) have = ((float)(e.y - e.x) >= sh.span) == (stage == 0);
                if (e.x >= bnd || e.y < a) {              // no element of the row in the slice
                    if (OBJ == ZL_OBJ_SUM && have && e.y < a) carry += e.y;
                    have = false;
                }
            }
            list_rows(list, sh.fill, packed, rd, R, row, have, e.x, e.y, a, bnd, sh.slack);
        }
        __syncthreads();
        const int rows = (int)(packed ? sh.fill.packed >> LIST_BITS : sh.fill.wide >> 40);
        const uint32_t pieces = packed ? sh.fill.packed & ((1u << LIST_BITS) - 1u) : (uint32_t)sh.fill.wide;
        if (rows > 0) stream_list(list, sh.more, rows, pieces, rd, R, a, bnd, [&](const uint32_t (&T)[9]) {
            if (OBJ == ZL_OBJ_RANGE) {
                // cell[k] becomes a lower bound of G at the start of cell k (before the prefix maximum): an element
                // says that G is at least its successor for the cells after its own.  Elements before the slice
                // count for its first cell; those in its last cell or behind it go to cell[m], which is not looked
                // at.  A gap of at most `gap` cannot push a cell's bound, G less the cell's end, beyond that: it discards no cell.
                uint32_t longer = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) longer = max(longer, T[j + 1] - T[j]);
                if (longer > gap) {
#pragma unroll
                    for (int h = 0; h < 8; h += 4) {
                        uint32_t k[4], v[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            k[j] = T[h + j] < a ? 0u : min(((T[h + j] - a) >> shift) + 1u, m);
                            v[j] = cell[k[j]];
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) if (T[h + j + 1] - T[h + j] > gap && v[j] < T[h + j + 1]) atomicMax(&cell[k[j]], T[h + j + 1]);
                    }
                }
            } else {
                uint32_t in = 0;
#pragma unroll
                for (int j = 1; j < 9; ++j) {
                    const uint32_t d = T[j] - a, delta = T[j] - T[j - 1];
                    if (d < w) { atomicAdd(cell + (d >> shift), delta); in += delta; }
                }
                total += in;
                if (T[0] < a && T[8] >= a) {              // the row's last element before the slice
                    uint32_t before = T[0];
#pragma unroll
                    for (int j = 1; j < 8; ++j) if (T[j] < a) before = T[j];
                    carry += before;
                }
            }
        });
        __syncthreads();
        if (tid == 0) { sh.fill.packed = 0; sh.fill.wide = 0; if (stage == 0) sh.took += pieces; }
    }
    if (OBJ == ZL_OBJ_SUM) {
        carry = warp_sum64(carry);
        total = warp_sum64(total);
        if (lane == 0) { atomicAdd(&sh.acc, (unsigned long long)carry); atomicAdd(&sh.total, (unsigned long long)total); }
    }
}

// Dynamic shared memory: the slice's cells [cap + 4] u32 | rows' first and last element, relative [n] uint2 | SUM: per 128
// cells the scan before them and the smallest lower bound among them [cap / 128] two u64 | one Answers (three in a cluster),
// over which the list of rows to look through lies.
template <int OBJ, class SRC, class FORM>
__global__ void __launch_bounds__(FORM::THREADS, 1) k_cells(const SRC src, const CellParams P) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ CellShared<OBJ, FORM> sh;
    constexpr bool ONE = FORM::ONE;
    typedef typename CellShared<OBJ, FORM>::Sum Sum;
    cg::cluster_group cl = cg::this_cluster();
    const int b = blockIdx.y, rank = ONE ? 0 : blockIdx.x, G = ONE ? 1 : gridDim.x;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int n = P.n, R = P.R;
    uint32_t *cell = (uint32_t *)smem;
    uint2 *ends = (uint2 *)(cell + P.cap + 4);
    uint64_t *blk_before = (uint64_t *)(ends + n), *blk_lb = blk_before + P.cap / 128;
    Answers<FORM::NODES> *answers = (Answers<FORM::NODES> *)(OBJ == ZL_OBJ_SUM ? blk_lb + P.cap / 128 : blk_before);
    // A CTA's shared memory may be written by the others only once it runs: everybody says so here, and waits for the rest
    // with the columns read, before the first store into another CTA.
    if (G > 1) cl.barrier_arrive();
    // What takes no input comes before the wait for the kernel in front.
#pragma unroll 1
    for (int c = tid; c <= P.cap / 4; c += nt) reinterpret_cast<uint4 *>(cell)[c] = make_uint4(0, 0, 0, 0);
    if (tid == 0) { sh.acc = 0; sh.total = 0; sh.ncells = 0; sh.later = 0; sh.slow = 0; sh.gap = 0; sh.nnodes = 0; sh.fill.packed = 0; sh.fill.wide = 0; }
    if (tid < CELL_BATCH) {
        sh.gmax[tid] = sh.heard[0].gmax[tid] = sh.heard[ONE ? 0 : 1].gmax[tid] = 0;
        sh.gmin[tid] = sh.heard[0].gmin[tid] = sh.heard[ONE ? 0 : 1].gmin[tid] = INF32;
    }
    for (int k = tid; k < GUARD_BINS; k += nt) sh.hist[k] = 0;
    grid_dep_wait();
    const int r0 = ONE ? 0 : min(rank * P.rpc, n), nrows = ONE ? n : min(P.rpc, n - r0);
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
            const int h = (R - 1) / 2;
            const bool probe = OBJ == ZL_OBJ_RANGE && R > 2 && (r0 + p) % step == 0;
            const int64_t x = row.at(0), y = row.at(R - 1), z = probe ? row.at(h) : 0;
            if (probe) {
                // RANGE, a few dozen rows: how far the row's middle element is from where a row of equal gaps has it, in gaps: after h of R - 1
                // gaps with a standard deviation of s (in gaps) that is s * sqrt(h * (R - 1 - h) / (R - 1)) on average
                const float span = (float)(y - x), off = (float)(z - x) * (float)(R - 1) - span * (float)h;
                if (span > 0.f) irr += off * off / (span * span) * ((float)(R - 1) / ((float)h * (float)(R - 1 - h)));
            }
            const uint64_t ux = (uint64_t)x ^ (1ull << 63), uy = (uint64_t)y ^ (1ull << 63);
            q[0] = min(q[0], ux); q[1] = max(q[1], ux); q[2] = min(q[2], uy); q[3] = max(q[3], uy);
            ends[r0 + p] = make_uint2((uint32_t)(uint64_t)x, (uint32_t)(uint64_t)y);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q[k] = (k & 1) ? warp_max64(q[k]) : warp_min64(q[k]);
            if (lane == 0) sh.red[k][warp] = q[k];
        }
        if (OBJ == ZL_OBJ_RANGE) {
            irr = warp_sum(irr);
            if (lane == 0) sh.keys[warp] = (uint64_t)__float_as_uint(irr);
        }
        __syncthreads();
        if (G > 1) {
            cl.barrier_wait();
#pragma unroll 1
            for (int r = 0; r < G; ++r) {
                if (r == rank) continue;
                uint2 *to = map_shared_rank<ONE>(ends, r);
#pragma unroll 1
                for (int p = tid; p < nrows; p += nt) to[r0 + p] = ends[r0 + p];
            }
        }
#pragma unroll 1
        for (int k = warp; k < (OBJ == ZL_OBJ_RANGE ? 5 : 4); k += nw) {
            if (k < 4) {
                uint64_t v = lane < nw ? sh.red[k][lane] : (k & 1) ? 0ull : ~0ull;
                v = (k & 1) ? warp_max64(v) : warp_min64(v);
                if (lane < G) map_shared_rank<ONE>(&sh, lane)->ex[k][rank] = v;
            } else {
                const float v = warp_sum(lane < nw ? __uint_as_float((uint32_t)sh.keys[lane]) : 0.f);
                if (lane < G) map_shared_rank<ONE>(&sh, lane)->exi[rank] = v;
            }
        }
    }
    auto sync_cluster = [&]() { if (G > 1) cl.sync(); else __syncthreads(); };      // (a cluster barrier of one CTA takes several times as long)
    if constexpr (!std::is_same<SRC, AriBatch>::value) if (P.check_sorted) {
        const bool bad = rows_unsorted(src.ts + ((size_t)b * n + r0) * R, nrows, R);
        const int any = __syncthreads_or(bad);
        if (tid < G) map_shared_rank<ONE>(&sh, tid)->exc[rank] = any ? 1ull : 0ull;
    }
    sync_cluster();
    int64_t tmin;
    {
    InstMeta M;
    {
        uint64_t q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q[k] = lane < G ? (uint64_t)sh.ex[k][lane] : (k & 1) ? 0ull : ~0ull;
            q[k] = (k & 1) ? warp_max64(q[k]) : warp_min64(q[k]);
        }
        tmin = (int64_t)(q[0] ^ (1ull << 63));
        const int64_t t0 = (int64_t)(q[1] ^ (1ull << 63));
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
        if (P.check_sorted && M.status == ZL_OK && __any_sync(FULL, lane < G && sh.exc[min(lane, G - 1)])) M.status = ZL_ERR_UNSORTED;
        M.cscale = M.status == ZL_OK && M.use32 ? 1u : 0u;
        if (rank == 0 && tid == 0) P.meta[b] = M;
    }
    if (!M.cscale) {                                              // the same in the whole cluster
        if (rank == 0 && tid == 0) {
            P.flags[2] = P.epoch;                                 // the last kernel writes this instance's outputs
            if (M.status == ZL_OK) P.flags[1] = P.flags[3] = P.epoch;
        }
        return;
    }
    if (tid == 0) { sh.tmin = M.tmin; sh.t0 = (uint32_t)M.t0; sh.lmin = (uint32_t)M.lmin; sh.tend = (uint32_t)M.tend; }
    }
    {
        uint32_t longest = 0;
        const uint32_t tminlo = (uint32_t)(uint64_t)tmin - 1u;
#pragma unroll 2
        for (int p = tid; p < n; p += nt) {
            uint2 e = ends[p];
            e.x -= tminlo; e.y -= tminlo;
            ends[p] = e;
            longest = max(longest, e.y - e.x);
        }
        longest = __reduce_max_sync(FULL, longest);
        if (lane == 0) sh.red[0][warp] = longest;
    }
    __syncthreads();
    if (OBJ == ZL_OBJ_RANGE) {
        // Guards: the rows that can set G near the optimum.  At a random time row i's next element is uniform in its mean
        // gap m_i away, so all are within x with probability prod(x / m_i) over the rows with m_i > x; the smallest d of
        // about N = n * R tries is the x where sum(log(m_i / x)) reaches log(N), and rows with gaps shorter than that
        // hardly matter.  With the rows counted by the logarithm of their span that is a prefix sum of a prefix sum.  Rows
        // a bin shorter are taken along, and more of them where single gaps are much longer than the row's mean.  (A fifth
        // to a half of the rows on the workloads at hand.  A fixed fifth leaves dozens of cells where single gaps are
        // long: n=1024, R=1024, B=64 87 us; a fixed half costs n=128, R=256, B=1024 68 us instead of 53.)
        const uint32_t longest = __reduce_max_sync(FULL, lane < nw ? (uint32_t)sh.red[0][lane] : 0u);
        const int top = __float_as_int((float)longest) >> 20;
#pragma unroll 2
        for (int p = tid; p < n; p += nt) {
            const uint2 e = ends[p];
            atomicAdd(&sh.hist[min(GUARD_BINS - 1, top - (__float_as_int((float)(e.y - e.x)) >> 20))], 1u);
        }
        __syncthreads();
        float span;
        {                                                         // every warp by itself
            const uint32_t x0 = sh.hist[2 * lane], x1 = sh.hist[2 * lane + 1];
            uint32_t inc = x0 + x1;                               // rows in the bins up to the lane's second one
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, inc, d); if (lane >= d) inc += y; }
            const uint32_t n0 = inc - x1, n1 = inc;               // rows up to bin 2 lane, 2 lane + 1
            uint32_t dep = n0 + n1;                               // sum of these over the bins: (bin - own bin) over the rows, from the next bin on
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) { const uint32_t y = __shfl_up_sync(FULL, dep, d); if (lane >= d) dep += y; }
            const uint32_t d0 = dep - n0 - n1, d1 = dep - n1;     // that sum at bin 2 lane, 2 lane + 1
            const uint32_t tries = (uint32_t)(8.f * log2f((float)n * (float)R)), least = (uint32_t)min(n, 8);
            const int at = __reduce_min_sync(FULL, d0 >= tries ? 2 * lane : d1 >= tries ? 2 * lane + 1 : GUARD_BINS);
            const float irr = warp_sum(lane < G ? sh.exi[min(lane, G - 1)] : 0.f);
            const float dev = sqrtf(irr / (float)((n + (n + 31) / 32 - 1) / ((n + 31) / 32)));
            int k = at + 1 + (int)(GUARD_IRREGULAR * max(0.f, min(1.f, dev) - 0.1f));
            k = max(k, __reduce_min_sync(FULL, n0 >= least ? 2 * lane : n1 >= least ? 2 * lane + 1 : GUARD_BINS));
            span = k >= min(GUARD_BINS - 1, top) ? 0.f : __int_as_float((top - k) << 20);
            if (tid == 0) {
                if (dev * sqrtf((float)R) > 2.f * CELL_OFF) sh.slow = 1;      // (dev * sqrt(R) / 2 elements in the middle)
                sh.span = span;
                sh.slack = CELL_SLACK + (P.near ? (int)min(32.f, 0.5f * dev * sqrtf((float)R)) : 0);
                // gaps that are shorter than the smallest d that is to be expected hardly matter
                sh.gap = at < GUARD_BINS && top - at > EXPECTED_BINS ? (uint32_t)(__int_as_float((top - at - EXPECTED_BINS) << 20) / (float)max(R - 1, 1)) : 0u;
                sh.width = R > 1 ? (float)longest / ((float)(R - 1) * RANGE_CELLS) : 0.f;
                sh.lo = 1; sh.hi = sh.lmin + 1u; sh.ub = ~0ull;
            }
        }
        float el = 0.f;
        const uint32_t lmin = sh.lmin;
#pragma unroll 2
        for (int p = tid; p < n; p += nt) {
            const float w = (float)(ends[p].y - ends[p].x);
            if (w < span) el += min(1.f, (float)(lmin - min(lmin, ends[p].x)) / w) * (float)R;
        }
        el = warp_sum(el);
        if (lane == 0) atomicAdd(&sh.later, (unsigned long long)el);
    } else {
        // the wait at one time between the last worker's start and the first row's end
        const uint32_t t0 = sh.t0, lm = max(sh.lmin, t0);
        {
            const uint32_t t = t0 + (lm - t0) / 2;
            const RowReader<SRC> rd(src, b, P.B, n, R, sh.tmin);
            uint64_t acc = 0;
#pragma unroll 1
            for (int p = tid; p < nrows; p += nt) {
                const uint2 e = ends[r0 + p];
                acc += t - rd.in(r0 + p, max(0, first_at_or_after(rd, r0 + p, R, t + 1u, e.x, e.y) - 1));
            }
            acc = warp_sum64(acc);
            if (lane == 0) atomicAdd(&sh.acc, (unsigned long long)acc);
        }
        unsigned long long *es = (unsigned long long *)answers;   // (64 words, not in use yet)
        if (tid < 64) es[tid] = 0;
        __syncthreads();
        if (tid < G) map_shared_rank<ONE>(&sh, tid)->exs[rank] = sh.acc;
        sync_cluster();
        const uint64_t ub = warp_sum64(lane < G ? (uint64_t)sh.exs[min(lane, G - 1)] : 0ull);
        // times past lm at which the exhausted rows alone wait longer than that are left out: the first of 32 trial times
        // where they do (closer together near lm), then the first of 32 more between that one and the one before it
        const uint32_t tend = sh.tend;
        uint32_t below = lm, stop = lm + (uint32_t)min(ub, (uint64_t)(tend - lm));
#pragma unroll 1
        for (int part = 0; part < 2; ++part, es += 32) {
            const uint64_t k = part ? 32ull * (lane + 1) : (uint64_t)((lane + 1) * (lane + 1));
            const uint32_t trial = below + (uint32_t)(((uint64_t)(stop - below) * k) >> 10);
            uint64_t e = 0;
#pragma unroll 4
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
        if (tid == 0) {
            sh.acc = 0;
            sh.lo = t0; sh.hi = max(t0, min(stop, tend)) + 1u; sh.ub = ub; sh.slack = CELL_SLACK; sh.span = 0.f;
            // n cell widths are the looseness of a cell's bounds; the wait itself spreads over time by about sqrt(n) times
            // 0.29 iterations, an iteration being about twice the mean wait of a worker.  (n=17, R=700, B=20: half the factor
            // 73 us, twice the factor 840, with six instances left over; n=32, R=400, B=20 41, 39 and 68.)
            sh.width = SUM_WIDTH * (float)ub / ((float)n * sqrtf((float)n));
        }
    }
    if (tid == 0) {
        // the cells, and the CTA's slice of them
        const uint32_t lo = sh.lo, hi = sh.hi;
        uint32_t shift = sh.width >= 2.f ? (uint32_t)min(31, (__float_as_int(sh.width) >> 23) - 127) : 0u;
        while (((hi - lo - 1u) >> shift) >= (uint32_t)(G * P.cap)) ++shift;
        const uint32_t ncells = ((hi - lo - 1u) >> shift) + 1u;
        const uint32_t per = ((ncells + G - 1) / G + 3u) & ~3u;   // cells of a CTA (cap is a multiple of 128, so they fit)
        const uint32_t c0 = min((uint32_t)rank * per, ncells), c1 = min(c0 + per, ncells);
        sh.shift = shift; sh.c0 = c0; sh.m = c1 - c0;
        sh.a = lo + (c0 << shift); sh.bnd = c1 == ncells ? hi : lo + (c1 << shift);
        // cells asked for at first: the most promising one of every CTA, as far as the answers cost the warps no second turn (one only
        // across the bus: n=274, R=1062, B=8 from the host 226 us with four, 212 with one)
        sh.firsts = P.near ? max(1, min(min(CELL_FIRST, G), nw / ((P.rpc + 31) >> 5))) : 1;
        // with a few cells on either side of it: SUM so many as give about a dozen answers
        sh.around = OBJ == ZL_OBJ_RANGE ? 1 : (int)max(2u, min(8u, (uint32_t)(8ull * ncells / ((unsigned long long)n * R))));
        sh.bd = ~0ull; sh.bt = INF32; sh.ndone = 0; sh.asked = 0; sh.took = 0;
    }
    __syncthreads();
    const int m = (int)sh.m, nblk = (m + 127) >> 7;
    bool fits = true;
    int stage = 0, streamed = -1, evaluated = 0;                  // RANGE: 0 the guards, 1 (seldom) the other rows too; evaluations
    auto done = [&](uint32_t c) { return sh.ndone != 0 && was_asked(sh.asked_run, sh.ndone, c); };      // seldom called: for a cell that would be evaluated (once more)
#pragma unroll 1
    for (int round = 0;; ++round) {                               // a round: the most promising cells are evaluated, the rest counted
        // ---- the rows' elements in the slice
        if (streamed != stage) look_through<OBJ, SRC, FORM>(sh, cell, answers, ends, src, P.B, n, R, stage);
        streamed = stage;
        // ---- what the sweep knows at every cell's start; a warp takes a run of 128-cell blocks, four cells a lane
        const int bpw = (nblk + nw - 1) / nw, k0 = min(warp * bpw, nblk), k1 = min(k0 + bpw, nblk);
        typedef typename std::conditional<OBJ == ZL_OBJ_RANGE, uint32_t, uint64_t>::type ST;
        {
            ST t = 0;
#pragma unroll 2
            for (int k = k0; k < k1; ++k) {
                const uint4 v = *reinterpret_cast<const uint4 *>(cell + 128 * k + 4 * lane);
                if constexpr (OBJ == ZL_OBJ_RANGE) t = max(max(t, max(v.x, v.y)), max(v.z, v.w));
                else t += (uint64_t)v.x + v.y + v.z + v.w;
            }
            if constexpr (OBJ == ZL_OBJ_RANGE) t = __reduce_max_sync(FULL, t); else t = warp_sum64(t);
            if (lane == 0) sh.red[0][warp] = t;
        }
        __syncthreads();
        uint64_t key = ~0ull, kbase = 0;
        const uint32_t a = sh.a, bnd = sh.bnd, shift = sh.shift, c0 = sh.c0;
        if constexpr (OBJ == ZL_OBJ_RANGE) {
            uint32_t run = max(sh.t0, __reduce_max_sync(FULL, lane < warp ? (uint32_t)sh.red[0][lane] : 0u));
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
                    if (c < m && g[j] != INF32 && q < key && !done(c0 + (uint32_t)c)) { key = q; kbase = g[j]; }
                }
            }
        } else {
            uint64_t run, all;
            {
                const uint64_t x = lane < nw ? (uint64_t)sh.red[0][lane] : 0ull;
                run = sh.acc + warp_sum64(lane < warp ? x : 0ull);
                all = warp_sum64(x);
            }
            const uint64_t nn = (uint64_t)n;
#pragma unroll 1
            for (int k = k0; k < k1; ++k) {
                const uint4 v = *reinterpret_cast<const uint4 *>(cell + 128 * k + 4 * lane);
                const uint64_t s1 = v.x, s2 = s1 + v.y, s3 = s2 + v.z, s4 = s3 + v.w;
                uint64_t inc = s4;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) { const uint64_t y = shfl_up(inc, d); if (lane >= d) inc += y; }
                const uint64_t before = run + inc - s4;
                const uint32_t c = 128u * k + 4u * lane, start = a + (c << shift);
                uint64_t lbm = ~0ull;
                if (s4 != 0) {
                    // four cells together: none has a wait below the bound of the first one's start and all their elements
                    const uint64_t l = nn * start > before + s4 ? nn * start - (before + s4) : 0ull;
                    lbm = l;
                    if (sh.ndone == 0) {
                        // ... and the last one with elements in it attains at most this
                        const uint32_t j = v.w ? 3u : v.z ? 2u : v.y ? 1u : 0u;
                        const uint64_t u = nn * cell_end(start + (j << shift), shift, bnd) - (before + s4);
                        const uint64_t q = min(u, (uint64_t)0xffffffffffull) << 24 | (c0 + c + j + 1u);
                        if (q < key) { key = q; kbase = before + s4 - (j == 3u ? v.w : j == 2u ? v.z : j == 1u ? v.y : v.x); }
                    } else {
                        const uint64_t S[4] = {before + s1, before + s2, before + s3, before + s4};
                        const uint32_t dv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint64_t u = nn * cell_end(start + ((uint32_t)j << shift), shift, bnd) - S[j];
                            const uint64_t q = min(u, (uint64_t)0xffffffffffull) << 24 | (c0 + c + (uint32_t)j + 1u);
                            if (dv[j] != 0u && q < key && !done(c0 + c + (uint32_t)j)) { key = q; kbase = S[j] - dv[j]; }
                        }
                    }
                }
                lbm = warp_min64(lbm);
                if (lane == 0) { blk_before[k] = run; blk_lb[k] = lbm; }
                run += shfl_idx(inc, 31);
            }
            // a cell's 32-bit sum wrapped around: nothing in the slice can be trusted
            if (all != sh.total) fits = false;
        }
        {
            const uint64_t mine = warp_min64(key);
            if (key == mine) { sh.keys[warp] = mine; sh.kbases[warp] = kbase; }     // (keys are different, but where there is none)
            __syncthreads();
            if (warp == 0) {
                if (lane == 0) sh.ncells = 0;                     // (written to by the others behind the next cluster barriers)
                const uint64_t x = lane < nw ? (uint64_t)sh.keys[lane] : ~0ull;
                const uint64_t k = warp_min64(x);
                uint64_t base = sh.kbases[__ffs(__ballot_sync(FULL, x == k)) - 1];
                uint32_t first = 0;
                if (k != ~0ull) {                                 // a few cells before it come along
                    const int c = (int)((uint32_t)(k & 0xffffffu) - 1u - c0), from = max(c - sh.around, 0);
                    first = c0 + (uint32_t)from;
                    if constexpr (OBJ == ZL_OBJ_RANGE) base = cell[from];
                    else base -= warp_sum64(lane < c - from ? (uint64_t)cell[min(from + lane, c)] : 0ull);
                }
                if (lane < G) {
                    auto &to = *map_shared_rank<ONE>(&sh, lane);
                    to.exv[rank] = fits ? k : 0ull;
                    to.exb[rank] = base;
                    to.exf[rank] = first;
                }
            }
        }
        sync_cluster();
        // ---- the most promising cells: the best one of each CTA, in their order
        int some = 0, listed = 0, from = 0;                       // runs of this evaluation; of the list (0: not made yet), and how many of them were evaluated
        {
            uint64_t x = lane < G ? (uint64_t)sh.exv[min(lane, G - 1)] : ~0ull;
            if (__any_sync(FULL, x == 0ull)) fits = false;
            if (!fits) break;
            const int firsts = sh.firsts, ndone = sh.ndone;
#pragma unroll 1
            for (; some < firsts; ++some) {
                const uint64_t k = warp_min64(x);
                if (k == ~0ull) break;
                if (x == k) {
                    x = ~0ull;
                    if (warp == 0) {
                        // with a few cells around it
                        const uint32_t c = (uint32_t)(k & 0xffffffu) - 1u, first = sh.exf[lane], last = min(c + (uint32_t)sh.around, (sh.hi - 1u - sh.lo) >> shift);
                        sh.asked_run[ndone + some] = make_uint2(first, last);
                        sh.ca[some] = sh.lo + (first << shift); sh.ce[some] = cell_end(sh.lo + (last << shift), shift, sh.hi); sh.cb[some] = sh.exb[lane];
                        // no cell's bound is below this: gaps of no more discard no cell
                        if (some == 0 && OBJ == ZL_OBJ_RANGE && round == 0) sh.gap = max(sh.gap, (uint32_t)(k >> 24));
                    }
                }
            }
            if (some == 0) {                                      // none that has not been evaluated
                if (round == 0) fits = false;
                break;
            }
        }
        bool again = false;
#pragma unroll 1
        for (;;) {
            // ---- exactly
            __syncthreads();
            if (tid == 0) { if (listed == 0) { sh.ndone += some; sh.asked += 8; } else sh.asked += some; }
            fits = evaluate_cells<OBJ, SRC, FORM>(sh, answers, ends, src, P.B, n, R, P.rpc, evaluated & 1, some) <= FORM::NODES;
            ++evaluated;
            if (!fits) break;
            const uint64_t d = sh.bd;
            const uint32_t cb = (sh.bt - sh.lo) >> shift;
            if (listed == 0) {
                // ---- the cells that may still hold a smaller one, or the same one earlier: only cells before the best one's
                const uint64_t limit = d < INF32 ? d << 24 | (cb + 1u) : ~0ull;      // RANGE: the best one's key, as of a cell whose bound is attained
                auto keep = [&](uint32_t c, Sum base, Sum l) {
                    // (far too many already: how many more does not matter, and every CTA has been told of the same ones)
                    if (*(volatile unsigned int *)&sh.ncells > (unsigned)CELL_HOPELESS || done(c)) return;
                    // every CTA gets the list
#pragma unroll 1
                    for (int r = 0; r < G; ++r) {
                        auto &to = *map_shared_rank<ONE>(&sh, r);
                        const unsigned pos = atomicAdd(&to.ncells, 1u);
                        if (pos < CELL_ALIVE) { to.cell[pos] = c; to.base[pos] = base; to.lb[pos] = l; }
                    }
                };
                if constexpr (OBJ == ZL_OBJ_RANGE) {
#pragma unroll 1
                    for (int c = 4 * tid; c < m; c += 4 * nt) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(cell + c);
                        const uint32_t g[4] = {v.x, v.y, v.z, v.w};
                        unsigned in = 0;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t end = cell_end(a + ((uint32_t)(c + j) << shift), shift, bnd);
                            const uint64_t q = (uint64_t)(g[j] > end ? g[j] - end : 0u) << 24 | (c0 + (uint32_t)(c + j) + 1u);
                            if (c + j < m && q < limit) in |= 1u << j;
                        }
#pragma unroll 1
                        for (; in; in &= in - 1u) {
                            const int j = __ffs(in) - 1;
                            const uint32_t x = j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w, end = cell_end(a + ((uint32_t)(c + j) << shift), shift, bnd);
                            keep(c0 + (uint32_t)(c + j), x, x > end ? x - end : 0u);
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
                        uint64_t S = blk_before[k] + inc - s4;
#pragma unroll 1
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t c = (uint32_t)(128 * k + 4 * lane + j), x = cell[c];
                            const uint64_t st = (uint64_t)n * (a + (c << shift)), l = st > S + x ? st - S - x : 0ull;
                            if (x != 0u && (l < d || (l == d && c0 + c < cb))) keep(c0 + c, (Sum)S, (Sum)l);
                            S += x;
                        }
                    }
                }
                sync_cluster();
                listed = (int)sh.ncells;
                if (listed == 0) break;
                if (OBJ == ZL_OBJ_RANGE && stage == 0 && sh.span > 0.f && listed > CELL_ALIVE) {      // the other rows may discard them
                    stage = 1;
                    again = true;                                 // (a cluster barrier follows before the list is written to again)
                    break;
                }
                if (listed > CELL_ALIVE) {                        // more than there is room for: the next best cells may discard them
                    fits = again = round < CELL_ROUNDS && listed <= CELL_HOPELESS;
                    break;
                }
#pragma unroll 1
                for (int k = tid; k < listed; k += nt) {          // in the order of time
                    const uint32_t c = sh.cell[k];
                    int at = 0;
#pragma unroll 4
                    for (int i = 0; i < listed; ++i) at += sh.cell[i] < c;
                    sh.order[at] = (unsigned short)k;
                }
                __syncthreads();
                if (warp == 0) {                                  // runs of them
                    int runs = 0;
#pragma unroll 1
                    for (int i0 = 0; i0 < listed; i0 += 32) {
                        const int i = i0 + lane, k = i < listed ? sh.order[i] : 0;
                        const uint32_t c = sh.cell[k], before = i > 0 && i < listed ? sh.cell[sh.order[i - 1]] : 0u;
                        const bool head = i < listed && (i == 0 || c - before > CELL_RUN<OBJ> / 2 + 1 || c / CELL_RUN<OBJ> != before / CELL_RUN<OBJ>);
                        const unsigned heads = __ballot_sync(FULL, head);
                        const int r = runs + __popc(heads & (FULL >> (31 - lane))) - 1;
                        if (head) { sh.run[r] = make_uint2(c, c); sh.run_base[r] = sh.base[k]; sh.run_lb[r] = ~0ull; }
                        __syncwarp();
                        if (i < listed) { atomicMax(&sh.run[r].y, c); atomicMin(&sh.run_lb[r], (unsigned long long)sh.lb[k]); }
                        __syncwarp();
                        runs += __popc(heads);
                    }
                    if (lane == 0) sh.runs = runs;
                }
                __syncthreads();
                listed = sh.runs;
                // asking every row for each of them, or looking through the other rows first?
                if (OBJ == ZL_OBJ_RANGE && stage == 0 && sh.span > 0.f && listed > CELL_FEW && (long long)listed * n * CELL_ASK > (long long)sh.later) {
                    stage = 1;
                    again = true;
                    break;
                }
#pragma unroll 1
                for (int k = tid; k < listed; k += nt) {          // most promising first, of equal ones the earliest
                    const uint64_t l = sh.run_lb[k];
                    int at = 0;
#pragma unroll 2
                    for (int i = 0; i < listed; ++i) at += sh.run_lb[i] < l || (sh.run_lb[i] == l && i < k);
                    sh.order[at] = (unsigned short)k;
                }
                __syncthreads();
            } else {
                from += some;
            }
            // ---- the next runs of the list
            if (from >= listed) break;
            {
                // (SUM: a cell whose bound does not exceed d nearly always has to be looked at; many answers a cell are compared with one another)
                const int batch = OBJ == ZL_OBJ_SUM ? CELL_BATCH : max(4, min(CELL_BATCH, 4 * nt / P.rpc));
                const int x = sh.order[from];
                if (sh.run_lb[x] > d || (sh.run_lb[x] == d && sh.run[x].x >= cb)) break;
                some = min(listed - from, max(4, min(batch, CELL_PAIRS / sh.per_cell)));
                if (tid < some) {
                    const int y = sh.order[from + tid];
                    sh.ca[tid] = sh.lo + (sh.run[y].x << shift); sh.ce[tid] = cell_end(sh.lo + (sh.run[y].y << shift), shift, sh.hi); sh.cb[tid] = sh.run_base[y];
                }
            }
        }
        if (!again) break;
    }
    // no CTA leaves while another may still write to its memory: everybody says here that it has done so for the last time
    if (G > 1) cl.barrier_arrive();
    const uint64_t d = sh.bd;
    // Rows that the route is not made for: many evaluations, rows that stand still, RANGE rows far off their estimates or far more of
    // them in one slice than its share.  The result is as good as any, but the handle's next calls are better off elsewhere.
    if (tid == 0 && (sh.slow || sh.asked > (OBJ == ZL_OBJ_RANGE ? CELL_ASKED_RANGE : CELL_ASKED_SUM) ||
                     (OBJ == ZL_OBJ_RANGE && G > 1 && streamed == 0 && 16ll * G * ((long long)sh.took - 2 * n) > 3ll * n * R)))
        P.flags[3] = P.epoch;
    // (a result above the wait known to be attained means rows that are not sorted: the sweep decides)
    if (!fits || d == ~0ull || d > sh.ub) {
        if (rank == 0 && tid == 0) {
            P.meta[b].overflow = 1;
            P.flags[1] = P.flags[2] = P.flags[3] = P.epoch;
        }
    } else {
        const uint32_t bar = sh.bt + (OBJ == ZL_OBJ_RANGE ? (uint32_t)d : 0u);      // relative
        if (rank == 0 && tid == 0) {
            P.wait[b] = (int64_t)d;
            P.barrier[b] = sh.tmin - 1 + (int64_t)bar;
            if (P.status) P.status[b] = ZL_OK;
        }
        // ---- the indices of the own rows: the last element not after the barrier
        const RowReader<SRC> rd(src, b, P.B, n, R, sh.tmin);
#pragma unroll 1
        for (int p = tid; p < nrows; p += nt) {
            const uint2 e = ends[r0 + p];
            P.idx[(size_t)b * n + r0 + p] = first_at_or_after(rd, r0 + p, R, bar + 1u, e.x, e.y) - 1;
        }
    }
    if (G > 1) cl.barrier_wait();
}

// ------------------------------------------------------------------------------ the kernels of the forms
// Modules of their own: a module is loaded whole when one of its kernels is first named, and the forms for many instances are named only for handles that make
// such calls, the checked ones only for handles that ask for checks (all in one: the first handle of a process 28 ms, 20 before the forms).
enum CellFormOf { FORM_CLUSTER, FORM_ALONE, FORM_THREE, FORM_FOUR, FORM_FIVE, FORM_SEVEN };
template <class SRC> using CellKernel = void (*)(const SRC, const CellParams);
CellKernel<MatBatch> cell_kernel_crowded(MatBatch, int form);         // RANGE; cells_crowded.cu
CellKernel<AriBatch> cell_kernel_crowded(AriBatch, int form);
CellKernel<MatBatch> cell_kernel_crowded_sum(MatBatch, int form);     // SUM; cells_crowded_sum.cu
CellKernel<AriBatch> cell_kernel_crowded_sum(AriBatch, int form);
CellKernel<MatChecked> cell_kernel_checked(int objective, int form);  // cells_checked.cu

#ifndef ZL_CELLS_KERNELS_ONLY      // (cells_crowded.cu, cells_crowded_sum.cu and cells_checked.cu take the search from here)
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
struct CellShape { int cluster, threads, form, cap; size_t smem; };

// What a form takes of an SM: most threads, shared memory that the kernel declares, and (`dynamic`) what lies behind the cells.
struct CellRoom { int threads; size_t fixed, dynamic; };
template <int OBJ, class FORM>
static CellRoom cell_room_t() {
    const size_t d = std::max((FORM::ONE ? 1 : 3) * sizeof(Answers<FORM::NODES>), sizeof(RowList<FORM::ROWS>));
    return CellRoom{FORM::THREADS, sizeof(CellShared<OBJ, FORM>), (d + 15) & ~(size_t)15};
}
static CellRoom cell_room(int objective, int form) {
    if (objective != ZL_OBJ_RANGE) {
        return form == FORM_CLUSTER ? cell_room_t<ZL_OBJ_SUM, CellCluster>() : form == FORM_THREE ? cell_room_t<ZL_OBJ_SUM, CellThreeSum>()
               : form == FORM_FOUR ? cell_room_t<ZL_OBJ_SUM, CellFourSum>() : cell_room_t<ZL_OBJ_SUM, CellAlone>();
    }
    switch (form) {
        case FORM_CLUSTER: return cell_room_t<ZL_OBJ_RANGE, CellCluster>();
        case FORM_THREE: return cell_room_t<ZL_OBJ_RANGE, CellThree>();
        case FORM_FOUR: return cell_room_t<ZL_OBJ_RANGE, CellFour>();
        case FORM_FIVE: return cell_room_t<ZL_OBJ_RANGE, CellFive>();
        case FORM_SEVEN: return cell_room_t<ZL_OBJ_RANGE, CellSeven>();
        default: return cell_room_t<ZL_OBJ_RANGE, CellAlone>();
    }
}

static CellShape cell_shape(int n, int R, int B, int objective, int num_sms) {
    CellShape s;
    // CTAs: as many as there are SMs, each with ten rows and a thousand timestamps at least (n=23, R=63, B=8 17 us
    // with one CTA an instance, 21 with two).  More than eight only for the largest instances, of which
    // few fill the GPU: as many as find room at once for every instance with an SM to each CTA (there is for 7 clusters of 16 and for 11
    // of 10; n=4096, R=4096, B=8 149 us with 10, 187 with 16 CTAs of half the size).
    s.cluster = 1;
    while (s.cluster < 8 && (long long)B * s.cluster * 2 <= num_sms && n / (s.cluster * 2) >= 10 && (long long)n * R >= 1024ll * 2 * s.cluster) s.cluster *= 2;
    if ((long long)n * R >= (1 << 22) && n >= 16 * CELL_CLUSTER && s.cluster == 8 && B <= 11) s.cluster = B <= 7 ? CELL_CLUSTER : 10;
    const long long ctas = (long long)B * s.cluster;
    // CTAs that share an SM.  Clusters do not fill the GPU to the last SM: with an SM to each CTA there is room for 33 of 4 and 15 of 8
    // (n=1286, R=136, B=16 46 us for two turns of clusters of 8, 32 with a cluster's CTAs two to an SM).
    const int sms = s.cluster <= 2 || s.cluster > 8 ? num_sms : s.cluster == 4 ? num_sms * 9 / 10 : num_sms * 13 / 16;
    const int share = (int)std::max<long long>(1, std::min<long long>(8, (ctas + sms - 1) / sms));
    const bool crowded = objective == ZL_OBJ_RANGE && share >= 3;
    auto cells_in = [&](int form, double kb) {                     // cells that leave room for the CTAs that share an SM in so much shared memory
        const CellRoom r = cell_room(objective, form);
        const double left = std::min(200.0, kb / std::min(r.threads / 128, share)) * 1024 - (double)r.fixed - 1024 - 8.0 * n - 64 - (double)r.dynamic;
        return std::max(2048, (int)(left / (objective == ZL_OBJ_RANGE ? 4.0 : 4.125)) & ~127);
    };
    // RANGE: the cells that two groups of equal workers need, of all the rows the most: about n / 6 an iteration of the slow ones (n=83, R=109, B=1177 58 us with
    // 19 to each of R, 38 with 35; n=128, R=150, B=1024 74 with 16, 43 with 24; n=325, R=66, B=1366 93 with 44, 124 with 31); others do with less, but single instances of few workers (n=28, R=302,
    // B=2129 95 us with 11, 440 with 9, where lists overflow).
    const double need = R * std::min(0.5 * RANGE_CELLS, 6.0 + n / 6.0), least_cells = (n < 48 ? 1.2 : 0.7) * need;
    // The form.  Eight CTAs an SM instead of seven where that saves a turn (n=124, R=20, B=1109 27 us with eight, 31 with seven; n=300, R=60, B=1150 53 /
    // 62; but B=1363, two turns of either, n=62, R=93 55 / 53; n=565, R=34, B=1180 163 / 118), with as many cells; large instances that take
    // several turns five of them, with more cells and no spills (n=74, R=200, B=1354 with long single gaps 63 / 70; n=117, R=338, B=1476 with stragglers 66 / 74, n=560, R=31, B=3431 215 / 231;
    // but one turn of seven, n=128, R=256, B=1024 50 / 37).
    auto turns = [&](int per_sm) { return (ctas + per_sm * num_sms - 1) / (per_sm * num_sms); };
    const long long N = (long long)n * R;
    s.form = s.cluster > 1 ? FORM_CLUSTER : share < 3 ? FORM_ALONE : !crowded ? (share == 3 ? FORM_THREE : share == 4 && N > 8192 ? FORM_FOUR : FORM_ALONE) : share == 3 ? FORM_THREE : share == 4 && N > 128 * 24 ? FORM_FOUR : share < 6 ? FORM_FIVE
             : turns(8) < turns(7) && n <= 384 && cells_in(FORM_FOUR, 196.0) >= least_cells ? FORM_FOUR : N >= 12288 && turns(7) > 1 ? FORM_FIVE : FORM_SEVEN;
    // threads: as many as an SM holds, whose registers CTAs get for four warps at a time
    s.threads = 128 * std::max(1, cell_room(objective, s.form).threads / 128 / share);
    const int per_thread = 32 * (objective == ZL_OBJ_RANGE ? 24 : 8);
    // no more than one to so many timestamps, but enough for the passes over the cells where a CTA has an SM to itself (n=24, R=60, B=1 15.2 us
    // with 128, 14.0 with 256; SUM n=100, R=150, B=1 21.7 with 256, 21.2 with 384)
    const int least = share > 1 ? 128 : objective == ZL_OBJ_RANGE ? 256 : 384;
    s.threads = (int)std::min<long long>(s.threads, std::max<long long>(least, 32 * (((long long)n * R / s.cluster + per_thread - 1) / per_thread)));
    // Cells an instance can use.  RANGE: RANGE_CELLS to an iteration of the slowest row, of which there are rarely more than
    // half R before the first row runs out.  SUM: see SUM_WIDTH, 6 to 12 sqrt(n) cells an iteration.  No more than lets the
    // CTAs of the call be resident together, as far as there are registers for them.
    // RANGE, where three CTAs and more share an SM: cells that are not needed cost more than the passes over them, because what shared memory
    // takes is gone from the L1 cache, past which the rows stream (n=218, R=213, B=700 78 us with 228 KB an SM in use, 61 with 196, 73
    // again when the cells are as few but the memory is asked for all the same).  So 164 KB where that holds the cells (n=50, R=165, B=1313 with
    // long single gaps 58 us, 65 with 196; not few workers: n=33, R=301, B=599 45 us with 164, 36 with 196), or 196, or 228 (predicted n=27, R=591, B=760 225
    // us with 196, 56 with 228).  Few workers, whose bounds are less alike, never need 50 to each of R (n=27, R=151, B=398 33 us, 31 with 19).
    double want = objective == ZL_OBJ_RANGE ? RANGE_CELLS * 0.5 * R : 12.0 * R * std::sqrt((double)n);
    if (crowded) want = std::min(want, R * (20.0 + n / 4.0));
    want = std::max(256.0, std::min(want, (double)(1 << 18)));
    double kb = 224.0;
    if (crowded) kb = n >= 48 && cells_in(s.form, 164.0) >= need ? 164.0 : cells_in(s.form, 196.0) >= least_cells ? 196.0 : n < 48 || cells_in(s.form, 228.0) >= least_cells ? 228.0 : 196.0;
    s.cap = std::min(cells_in(s.form, kb), ((int)(want / s.cluster) + 127) & ~127);
    s.cap = std::max(256, s.cap);
    s.smem = (size_t)s.cap * 4 + 16 + (size_t)n * 8 + (objective == ZL_OBJ_RANGE ? 0 : (size_t)s.cap / 8) + cell_room(objective, s.form).dynamic;
    return s;
}

template <int OBJ, class SRC>
static CellKernel<SRC> cell_kernel(int form) {
    if constexpr (std::is_same<SRC, MatChecked>::value) return cell_kernel_checked(OBJ, form);
    else if (form == FORM_CLUSTER) return k_cells<OBJ, SRC, CellCluster>;
    else if (form == FORM_ALONE) return k_cells<OBJ, SRC, CellAlone>;
    else if constexpr (OBJ == ZL_OBJ_SUM) return cell_kernel_crowded_sum(SRC(), form);
    else return cell_kernel_crowded(SRC(), form);
}

template <int OBJ, class SRC>
static void enqueue_cells_t(const Pipeline &q, const FilterBufs &fb, const LaunchPlan &p, cudaStream_t st, cudaEvent_t *ev, const SRC &src) {
    const CellShape s = cell_shape(q.n, q.R, q.B, OBJ, q.num_sms);
    CellParams P;
    P.n = q.n; P.R = q.R; P.B = q.B;
    P.cap = s.cap; P.rpc = (q.n + s.cluster - 1) / s.cluster; P.check_sorted = (q.flags & ZL_FLAG_CHECK_SORTED) ? 1 : 0;
    P.near = q.cells != 2;
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
    if (q.cells != 3) {
        launch(cell_kernel<OBJ, SRC>(s.form), dim3(s.cluster, q.B), s.threads, s.smem, s.cluster, src, P);
    }
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
    launch(k_cell_rest<OBJ, decltype(plain_rows(src))>, dim3((unsigned)std::max<long long>(1, std::min<long long>(q.num_sms, items))), CELL_REST_THREADS, p.smem, 1, plain_rows(src), sp, P, f);
    if (ev) cudaEventRecord(ev[4], st);
}

void enqueue_cells(const Pipeline &q, const FilterBufs &fb, const LaunchPlan &p, cudaStream_t st, cudaEvent_t *ev, const MatBatch &src) {
    const MatChecked checked{src.ts, q.guard};
    if (q.guard) {
        if (q.objective == ZL_OBJ_RANGE) enqueue_cells_t<ZL_OBJ_RANGE>(q, fb, p, st, ev, checked); else enqueue_cells_t<ZL_OBJ_SUM>(q, fb, p, st, ev, checked);
    } else if (q.objective == ZL_OBJ_RANGE) {
        enqueue_cells_t<ZL_OBJ_RANGE>(q, fb, p, st, ev, src);
    } else {
        enqueue_cells_t<ZL_OBJ_SUM>(q, fb, p, st, ev, src);
    }
}
void enqueue_cells(const Pipeline &q, const FilterBufs &fb, const LaunchPlan &p, cudaStream_t st, cudaEvent_t *ev, const AriBatch &src) {
    if (q.objective == ZL_OBJ_RANGE) enqueue_cells_t<ZL_OBJ_RANGE>(q, fb, p, st, ev, src); else enqueue_cells_t<ZL_OBJ_SUM>(q, fb, p, st, ev, src);
}

template <int OBJ, class SRC>
static cudaError_t cell_limits_t(bool crowded) {
    const int big = 200 * 1024;
    auto raise = [&](auto kernel) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
        return e == cudaSuccess ? cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : e;
    };
    cudaError_t e = cudaSuccess;
    if (crowded) {
        for (int form : {FORM_THREE, FORM_FOUR, FORM_FIVE, FORM_SEVEN})
            if (e == cudaSuccess && (OBJ == ZL_OBJ_RANGE || form <= FORM_FOUR)) e = raise(cell_kernel<OBJ, SRC>(form));
        return e;
    }
    for (int form : {FORM_CLUSTER, FORM_ALONE}) if (e == cudaSuccess) e = raise(cell_kernel<OBJ, SRC>(form));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cell_rest<OBJ, decltype(plain_rows(std::declval<SRC>()))>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
    return e;
}

cudaError_t cell_limits() {
    cudaError_t e = cell_limits_t<ZL_OBJ_RANGE, MatBatch>(false);
    if (e == cudaSuccess) e = cell_limits_t<ZL_OBJ_RANGE, AriBatch>(false);
    if (e == cudaSuccess) e = cell_limits_t<ZL_OBJ_SUM, MatBatch>(false);
    if (e == cudaSuccess) e = cell_limits_t<ZL_OBJ_SUM, AriBatch>(false);
    return e;
}
bool cell_crowded(int B, int num_sms) { return B > 2 * num_sms; }
cudaError_t cell_crowded_limits(int objective) {
    const bool sum = objective != ZL_OBJ_RANGE;
    const cudaError_t e = sum ? cell_limits_t<ZL_OBJ_SUM, MatBatch>(true) : cell_limits_t<ZL_OBJ_RANGE, MatBatch>(true);
    return e != cudaSuccess ? e : sum ? cell_limits_t<ZL_OBJ_SUM, AriBatch>(true) : cell_limits_t<ZL_OBJ_RANGE, AriBatch>(true);
}
cudaError_t cell_checked_limits() {
    cudaError_t e = cell_limits_t<ZL_OBJ_RANGE, MatChecked>(false);
    if (e == cudaSuccess) e = cell_limits_t<ZL_OBJ_RANGE, MatChecked>(true);
    return e == cudaSuccess ? cell_limits_t<ZL_OBJ_SUM, MatChecked>(false) : e;
}

#endif

}  // namespace zl
