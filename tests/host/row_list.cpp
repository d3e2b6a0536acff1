// One CTA's reading of rows, as the cell route does it, on the CPU.  ROWS_FILE and LOOK_FILE are cut out of the kernel's source.
#include "warp_on_cpu.h"

enum { ZL_OBJ_RANGE = 0, ZL_OBJ_SUM = 1 };
struct MatBatch { const int64_t *ts; };
struct AriBatch { const int64_t *last, *iv; };
static constexpr uint32_t INF32 = 0xffffffffu;
static inline uint64_t shfl_up(uint64_t v, int d) { return __shfl_up_sync(FULL, v, d); }
static inline uint64_t shfl_idx(uint64_t v, int i) { return __shfl_sync(FULL, v, i); }

#include ROWS_FILE

template <int ROWS_> struct Form { static constexpr int ROWS = ROWS_, NODES = 2048; };   // (NODES: room for the list)
template <int NODES> struct Answers { uint64_t words[NODES]; };
template <int OBJ, class FORM>
struct CellShared {
    int64_t tmin;
    uint32_t a, bnd, shift, gap, m, took;
    float span;
    int slack;
    ListFill fill;
    unsigned long long acc, total;
    uint32_t more[2][FORM::ROWS / 32];
};

#include LOOK_FILE

static void rows_are(const int64_t *ts, long long elements) { cpu::first = ts; cpu::end = ts + elements; cpu::bad = cpu::worst = 0; }
static long verdict(int64_t *worst) { *worst = cpu::worst; return cpu::bad; }

template <int OBJ, class FORM>
static void look_t(const MatBatch &src, int B, int n, int R, int64_t tmin, const uint32_t *ends, uint32_t a, uint32_t bnd, uint32_t shift, uint32_t m, uint32_t gap, float span,
                   int slack, int stage, int threads, uint32_t *cell, uint64_t *sums) {
    static CellShared<OBJ, FORM> sh;
    static Answers<FORM::NODES> answers[3];
    memset(&sh, 0, sizeof sh);
    sh.tmin = tmin; sh.a = a; sh.bnd = bnd; sh.shift = shift; sh.gap = gap; sh.m = m; sh.span = span; sh.slack = slack;
    cpu::run(threads, [&] { look_through<OBJ, MatBatch, FORM>(sh, cell, answers, (const uint2 *)ends, src, B, n, R, stage); });
    sums[0] = sh.acc; sums[1] = sh.total;
}

// A slice [a, bnd) of instance b in cells of 2^shift: what look_through makes of it with `threads` threads and lists of `rows` rows.
// Returns the number of loads from outside the matrix.
extern "C" long look(int objective, int rows, const int64_t *ts, int B, int n, int R, int b, int64_t tmin, const uint32_t *ends, uint32_t a, uint32_t bnd, uint32_t shift, uint32_t m,
                     uint32_t gap, float span, int slack, int stage, int threads, uint32_t *cell, uint64_t *sums, int64_t *worst) {
    rows_are(ts, (long long)B * n * R);
    blockIdx.y = b;
    auto *f = objective == ZL_OBJ_RANGE ? rows == 256 ? look_t<ZL_OBJ_RANGE, Form<256>> : rows == 512 ? look_t<ZL_OBJ_RANGE, Form<512>> : look_t<ZL_OBJ_RANGE, Form<1024>>
                                        : rows == 256 ? look_t<ZL_OBJ_SUM, Form<256>> : rows == 512 ? look_t<ZL_OBJ_SUM, Form<512>> : look_t<ZL_OBJ_SUM, Form<1024>>;
    f(MatBatch{ts}, B, n, R, tmin, ends, a, bnd, shift, m, gap, span, slack, stage, threads, cell, sums);
    return verdict(worst);
}

// The first element at or after t of a row, for each of `count` (row, t).
extern "C" long places(const int64_t *ts, int B, int n, int R, int b, int64_t tmin, const uint32_t *ends, int count, const int *row, const uint32_t *t, int *at, int64_t *worst) {
    rows_are(ts, (long long)B * n * R);
    const RowReader<MatBatch> rd(MatBatch{ts}, b, B, n, R, tmin);
    for (int i = 0; i < count; ++i) at[i] = first_at_or_after(rd, row[i], R, t[i], ends[2 * row[i]], ends[2 * row[i] + 1]);
    return verdict(worst);
}

extern "C" long unsorted(const int64_t *ts, int rows, int R, int threads, int *any, int64_t *worst) {
    rows_are(ts, (long long)rows * R);
    *any = 0;
    cpu::run(threads, [&] { if (rows_unsorted(ts, rows, R)) *any = 1; });
    return verdict(worst);
}
