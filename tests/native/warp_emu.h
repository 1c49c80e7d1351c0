// Runs the text of a kernel on the host: the threads of one block are fibers, a
// seeded scheduler picks the next one wherever a thread reaches a collective
// operation, so that a thread may run ahead of its warp as far as CUDA's model
// lets it. Threads of a warp that wait at different collectives end the run
// with exit code 3. Votes, shuffles and matches exchange values and order
// nothing: atomics whose results only others read may be held back
// (emu::defer_or) until the thread's next __syncwarp or __syncthreads.
#pragma once
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <random>
#include <vector>

#include <sys/mman.h>
#include <ucontext.h>

#define __global__
#define __device__
#define __host__
#define __forceinline__ inline
#define __launch_bounds__(...)
#define __align__(n) __attribute__((aligned(n)))
#define __shared__ static
#define __restrict__

struct Dim {
    unsigned x = 1, y = 1, z = 1;
};
struct uint4 {
    uint32_t x, y, z, w;
};
struct int4 {
    int32_t x, y, z, w;
};

using std::max;
using std::min;
inline uint64_t min(uint64_t a, unsigned long long b) { return a < b ? a : (uint64_t)b; }
inline uint64_t min(unsigned long long a, uint64_t b) { return a < b ? (uint64_t)a : b; }

namespace emu {

typedef unsigned __int128 Word;
enum Kind { kNone, kSyncwarp, kShfl, kShflUp, kShflDown, kShflXor, kBallot, kMatch, kRedMax, kRedMin, kRedAdd, kRedOr, kBlock };

struct Thread {
    ucontext_t ctx;
    Dim tid;
    bool done = false;
    Kind at = kNone;  // waiting there
    Word in = 0, out = 0;
    int arg = 0;
    unsigned syncs = 0;  // __syncwarp and __syncthreads passed
    std::vector<std::pair<unsigned long long*, unsigned long long>> held;  // deferred ORs
};

inline std::vector<Thread> threads;
inline Thread* cur = nullptr;
inline ucontext_t sched;
inline Dim block_dim, grid_dim, block_idx;
inline bool defer_or = false;
inline std::function<void()> body;
constexpr size_t kStack = 1u << 17;

inline void settle(Thread& t) {
    for (auto& h : t.held) *h.first |= h.second;
    t.held.clear();
}

inline Word wait(Kind k, Word in, int arg = 0) {
    Thread* const t = cur;
    if (k == kSyncwarp || k == kBlock) settle(*t);
    t->at = k;
    t->in = in;
    t->arg = arg;
    swapcontext(&t->ctx, &sched);
    if (k == kSyncwarp || k == kBlock) ++t->syncs;
    return t->out;
}

// the results of a collective that threads [lo, hi) all wait at
inline void complete(int lo, int hi) {
    const Kind k = threads[lo].at;
    const int n = hi - lo;
    Word all = 0;
    if (k == kRedMin) all = ~(Word)0;
    for (int i = lo; i < hi; ++i) {
        const Word x = threads[i].in;
        if (k == kBallot) all |= x ? (Word)1 << (i - lo) : 0;
        if (k == kRedMax) all = std::max(all, x);
        if (k == kRedMin) all = std::min(all, x);
        if (k == kRedAdd || k == kBlock) all += x;
        if (k == kRedOr) all |= x;
    }
    for (int i = lo; i < hi; ++i) {
        Thread& t = threads[i];
        int src = i - lo;
        if (k == kShfl) src = t.arg & 31;
        if (k == kShflUp && src >= t.arg) src -= t.arg;
        if (k == kShflDown && src + t.arg < n) src += t.arg;
        if (k == kShflXor) src ^= t.arg;
        t.out = k >= kShfl && k <= kShflXor ? threads[lo + src].in : all;
        if (k == kMatch) {
            t.out = 0;
            for (int j = lo; j < hi; ++j)
                if (threads[j].in == t.in) t.out |= (Word)1 << (j - lo);
        }
    }
    for (int i = lo; i < hi; ++i) threads[i].at = kNone;
}

inline void entry() {
    body();
    settle(*cur);
    cur->done = true;
    swapcontext(&cur->ctx, &sched);
}

// one block of n threads (a multiple of 32) running f
inline void run(unsigned n, unsigned block, unsigned grid, unsigned seed, std::function<void()> f) {
    std::mt19937 rng(seed);
    body = std::move(f);
    block_dim.x = n;
    block_idx.x = block;
    grid_dim.x = grid;
    threads = std::vector<Thread>(n);
    char* const stacks = (char*)mmap(nullptr, n * kStack, PROT_READ | PROT_WRITE,
                                     MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    for (unsigned i = 0; i < n; ++i) {
        Thread& t = threads[i];
        t.tid.x = i;
        t.tid.y = t.tid.z = 0;
        getcontext(&t.ctx);
        t.ctx.uc_stack.ss_sp = stacks + i * kStack;
        t.ctx.uc_stack.ss_size = kStack;
        t.ctx.uc_link = &sched;
        makecontext(&t.ctx, entry, 0);
    }
    std::vector<unsigned> ready(n);
    for (;;) {
        ready.clear();
        for (unsigned i = 0; i < n; ++i)
            if (!threads[i].done && threads[i].at == kNone) ready.push_back(i);
        if (ready.empty()) {  // everyone waits: complete what is complete
            bool moved = false, alive = false;
            unsigned at_block = 0, left = 0;
            for (unsigned w = 0; w < n; w += 32) {
                bool same = true;
                unsigned here = 0;
                for (unsigned i = w; i < w + 32; ++i) {
                    left += !threads[i].done;
                    here += !threads[i].done;
                    at_block += threads[i].at == kBlock;
                    same = same && !threads[i].done && threads[i].at == threads[w].at;
                }
                alive = alive || here;
                if (same && threads[w].at != kBlock) {
                    complete(w, w + 32);
                    moved = true;
                }
            }
            if (!alive) break;
            if (!moved && at_block == left && left == n) {
                complete(0, n);
                moved = true;
            }
            if (!moved) {
                fprintf(stderr, "threads of a warp wait at different collectives\n");
                exit(3);
            }
            continue;
        }
        std::shuffle(ready.begin(), ready.end(), rng);
        for (const unsigned i : ready) {
            cur = &threads[i];
            swapcontext(&sched, &cur->ctx);
        }
    }
    munmap(stacks, n * kStack);
}

template <class T>
Word word(T x) {
    Word w = 0;
    memcpy(&w, &x, sizeof(T));
    return w;
}
template <class T>
T value(Word w) {
    T x;
    memcpy(&x, &w, sizeof(T));
    return x;
}

}  // namespace emu

#define threadIdx (emu::cur->tid)
#define blockIdx emu::block_idx
#define blockDim emu::block_dim
#define gridDim emu::grid_dim

constexpr unsigned kFull = 0xFFFFFFFFu;
typedef unsigned __int128 u128;

inline void __syncwarp(unsigned = kFull) { emu::wait(emu::kSyncwarp, 0); }
inline void __syncthreads() { emu::wait(emu::kBlock, 0); }
inline int __syncthreads_count(int p) { return (int)emu::wait(emu::kBlock, p != 0); }
template <class T> T __shfl_sync(unsigned, T v, int l) { return emu::value<T>(emu::wait(emu::kShfl, emu::word(v), l)); }
template <class T> T __shfl_up_sync(unsigned, T v, int d) { return emu::value<T>(emu::wait(emu::kShflUp, emu::word(v), d)); }
template <class T> T __shfl_down_sync(unsigned, T v, int d) { return emu::value<T>(emu::wait(emu::kShflDown, emu::word(v), d)); }
template <class T> T __shfl_xor_sync(unsigned, T v, int d) { return emu::value<T>(emu::wait(emu::kShflXor, emu::word(v), d)); }
inline unsigned __ballot_sync(unsigned, int p) { return (unsigned)emu::wait(emu::kBallot, p != 0); }
inline int __any_sync(unsigned, int p) { return emu::wait(emu::kBallot, p != 0) != 0; }
inline unsigned __match_any_sync(unsigned, uint32_t x) { return (unsigned)emu::wait(emu::kMatch, x); }
inline unsigned __reduce_max_sync(unsigned, uint32_t x) { return (unsigned)emu::wait(emu::kRedMax, x); }
inline unsigned __reduce_min_sync(unsigned, uint32_t x) { return (unsigned)emu::wait(emu::kRedMin, x); }
inline unsigned __reduce_add_sync(unsigned, uint32_t x) { return (unsigned)emu::wait(emu::kRedAdd, x); }
inline unsigned __reduce_or_sync(unsigned, uint32_t x) { return (unsigned)emu::wait(emu::kRedOr, x); }

inline int __popc(uint32_t x) { return __builtin_popcount(x); }
inline int __ffs(uint32_t x) { return __builtin_ffs((int)x); }
inline int __ffsll(long long x) { return __builtin_ffsll(x); }
inline unsigned lanemask_lt() { return (1u << (threadIdx.x & 31)) - 1u; }
inline uint32_t __float_as_uint(float f) { return emu::value<uint32_t>(emu::word(f)); }
template <class T> T __ldg(const T* p) { return *p; }
template <class T> T __ldcg(const T* p) { return *p; }
template <class T> T __ldcs(const T* p) { return *p; }
template <class T, class U> T atomicAdd(T* p, U v) { const T o = *p; *p = (T)(o + (T)v); return o; }
template <class T, class U> T atomicSub(T* p, U v) { const T o = *p; *p = (T)(o - (T)v); return o; }
template <class T, class U> T atomicMin(T* p, U v) { const T o = *p; *p = std::min(o, (T)v); return o; }
template <class T> T atomicCAS(T* p, T c, T v) { const T o = *p; if (o == c) *p = v; return o; }
inline uint32_t atomicOr(uint32_t* p, uint32_t v) { const uint32_t o = *p; *p |= v; return o; }
inline unsigned long long atomicOr(unsigned long long* p, unsigned long long v) {
    const unsigned long long o = *p;
    if (emu::defer_or) emu::cur->held.push_back({p, v});
    else *p |= v;
    return o;
}
