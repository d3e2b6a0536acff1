// The few CUDA names that the row reading of the cell route uses, for one CTA on the CPU: every thread is a coroutine, which gives
// way wherever it waits for its warp or its CTA.  Loads from the rows are checked against the matrix; a bad one is counted and
// gives 0.
#pragma once
#include <ucontext.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <type_traits>
#include <vector>

using std::max;
using std::min;

#define __device__
#define __forceinline__ inline
#define __noinline__

struct uint2 { uint32_t x, y; };
static inline uint2 make_uint2(uint32_t x, uint32_t y) { return uint2{x, y}; }
struct Dim { int x = 0, y = 0; };
static Dim threadIdx, blockIdx, blockDim;

namespace cpu {

struct Thread { ucontext_t at; std::vector<char> stack; bool done = false; };
static std::vector<Thread> threads;
static ucontext_t home;
static int current;
static std::function<void()> body;
struct Meeting { int arrived = 0; long round = 0; };
static std::vector<Meeting> warps;
static Meeting block;
static std::vector<uint64_t> words[2];       // what the threads of a warp hand to one another, by turns

static void give_way() {
    Thread &t = threads[current];
    swapcontext(&t.at, &home);
}
static void meet(Meeting &m, int n) {
    const long r = m.round;
    if (++m.arrived == n) { m.arrived = 0; ++m.round; return; }
    while (m.round == r) give_way();
}
// the 32 values of the warp's threads
static const uint64_t *exchange(uint64_t v) {
    Meeting &w = warps[current >> 5];
    uint64_t *to = words[w.round & 1].data() + (current & ~31);
    to[current & 31] = v;
    meet(w, 32);
    return to;
}
static void entry() {
    body();
    threads[current].done = true;
    give_way();
}
static void run(int n, std::function<void()> f) {
    body = f;
    threads = std::vector<Thread>(n);
    warps.assign(n / 32, Meeting());
    block = Meeting();
    words[0].assign(n, 0); words[1].assign(n, 0);
    blockDim.x = n;
    for (Thread &t : threads) {
        t.stack.resize(64 << 10);
        getcontext(&t.at);
        t.at.uc_stack.ss_sp = t.stack.data(); t.at.uc_stack.ss_size = t.stack.size(); t.at.uc_link = nullptr;
        makecontext(&t.at, entry, 0);
    }
    for (int left = n; left > 0;) {
        for (current = 0; current < n; ++current) {
            if (threads[current].done) continue;
            threadIdx.x = current;
            swapcontext(&home, &threads[current].at);
            left -= threads[current].done;
        }
    }
}

// the rows
static const int64_t *first, *end;
static long bad;
static int64_t worst;                        // of the bad ones, the largest distance from the matrix in timestamps
static int64_t load(const int64_t *p) {
    if (p >= first && p < end) return *p;
    ++bad;
    worst = max(worst, (int64_t)(p >= end ? p - end + 1 : first - p));
    return 0;
}

}  // namespace cpu

static inline int64_t ldg64(const int64_t *p) { return cpu::load(p); }
static inline void load4(uint64_t &a, uint64_t &b, uint64_t &c, uint64_t &d, const int64_t *p) {
    if ((uintptr_t)p & 31) ++cpu::bad;       // 32 bytes on a 32-byte boundary
    a = ldg64(p); b = ldg64(p + 1); c = ldg64(p + 2); d = ldg64(p + 3);
}
static inline void prefetched(const int64_t *p) { cpu::load(p); }

static constexpr unsigned FULL = 0xffffffffu;
static inline void __syncthreads() { cpu::meet(cpu::block, blockDim.x); }
static inline void __syncwarp() { cpu::exchange(0); }
static inline int __popc(unsigned x) { return __builtin_popcount(x); }
static inline int __ffs(unsigned x) { return __builtin_ffs((int)x); }
template <class T> static T __shfl_sync(unsigned, T v, int from) { uint64_t w = 0; memcpy(&w, &v, sizeof v); w = cpu::exchange(w)[from & 31]; memcpy(&v, &w, sizeof v); return v; }
template <class T> static T __shfl_up_sync(unsigned m, T v, int d) { const int lane = threadIdx.x & 31; return __shfl_sync(m, v, lane >= d ? lane - d : lane); }
template <class T> static T __shfl_xor_sync(unsigned m, T v, int d) { return __shfl_sync(m, v, (threadIdx.x & 31) ^ d); }
static inline unsigned __ballot_sync(unsigned, bool p) { const uint64_t *w = cpu::exchange(p); unsigned r = 0; for (int i = 0; i < 32; ++i) r |= (unsigned)w[i] << i; return r; }
static inline uint32_t __reduce_or_sync(unsigned, uint32_t v) { const uint64_t *w = cpu::exchange(v); uint32_t r = 0; for (int i = 0; i < 32; ++i) r |= (uint32_t)w[i]; return r; }
static inline uint32_t __reduce_add_sync(unsigned, uint32_t v) { const uint64_t *w = cpu::exchange(v); uint32_t r = 0; for (int i = 0; i < 32; ++i) r += (uint32_t)w[i]; return r; }
static inline uint32_t __reduce_min_sync(unsigned, uint32_t v) { const uint64_t *w = cpu::exchange(v); uint32_t r = FULL; for (int i = 0; i < 32; ++i) r = min(r, (uint32_t)w[i]); return r; }
static inline uint32_t __reduce_max_sync(unsigned, uint32_t v) { const uint64_t *w = cpu::exchange(v); uint32_t r = 0; for (int i = 0; i < 32; ++i) r = max(r, (uint32_t)w[i]); return r; }
template <class T, class U> static T atomicAdd(T *p, U v) { const T was = *p; *p += (T)v; return was; }
template <class T, class U> static T atomicOr(T *p, U v) { const T was = *p; *p |= (T)v; return was; }
template <class T, class U> static T atomicMax(T *p, U v) { const T was = *p; *p = max(*p, (T)v); return was; }
template <class T, class U> static T atomicMin(T *p, U v) { const T was = *p; *p = min(*p, (T)v); return was; }
