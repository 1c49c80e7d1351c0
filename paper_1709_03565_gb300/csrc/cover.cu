// Coverage counting and the SKIS estimator (Sec. IV, Eq. 21, Alg. 2) and
// greedy max-coverage (Sec. V-A, Alg. 3, Eq. margin) on the device sketch.
//
// Coverage: each query of a batch of up to 64 owns one bit of a per-vertex
// mask. A small sketch is scanned in groups of 1 to 32 consecutive samples
// (k_coverage): a warp spreads a group's members over its lanes, ORs the
// members' masks per sample in shared memory and counts, per query bit, the
// samples whose OR has it (ballot + popcount). A large one is scanned in
// sample-id order (k_scan_ordered), and one with an inverted index by the
// seeds' sample lists (k_cover_inv). Counts and the estimator numerator are
// exact integers.
//
// Greedy: an inverted index vertex -> samples (counting sort), marginal
// coverage Delta_v, then per round an exact argmax of the integer key
// Delta_v W + T (2^f - w_v) (ties to the lowest id), and the samples of the
// chosen vertex are marked covered and their members' Delta decremented.
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <memory>
#include <new>
#include <string>

#include "../../include/skis.h"
#include "skis_internal.cuh"

namespace skis {

constexpr int kCovThreads = 256;
constexpr int kCovBlocks = 8;  // an SM: every warp slot
constexpr int kFillRuns = 4;  // k_fill_inverted

// Calls f(owner_lane, member) for every member of the samples held by the
// lanes (lane i: arena offset off, length len), spread over the warp: the
// members laid end to end, kRuns runs of 32 a pass with their loads in flight
// together, each lane finding the sample that holds its member by a search of
// the prefix sums.
template <int kRuns = 2, class F>
__device__ __forceinline__ void warp_members(uint64_t off, uint32_t len, const int32_t* __restrict__ arena, F&& f) {
    const int lane = threadIdx.x & 31;
    uint64_t sum = len;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint64_t y = __shfl_up_sync(kFull, sum, d);
        if (lane >= d) sum += y;
    }
    const uint64_t all = __shfl_sync(kFull, sum, 31);
    if (all >= (1ull << 32) - 32 * kRuns) {  // past 32-bit places: one sample after another
        for (int o = 0; o < 32; ++o) {
            const uint64_t o_off = __shfl_sync(kFull, off, o);
            const uint32_t o_len = __shfl_sync(kFull, len, o);
            for (uint64_t i = lane; i < o_len; i += 32) f(o, arena[o_off + i]);
        }
        return;
    }
    const uint32_t incl = (uint32_t)sum, total = (uint32_t)all;
    const uint64_t rel = off - (incl - len);  // + a member's place: its arena position
    for (uint32_t base = 0; base < total; base += 32 * kRuns) {
        int own[kRuns];
        int32_t u[kRuns];
#pragma unroll
        for (int k = 0; k < kRuns; ++k) own[k] = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1)
#pragma unroll
            for (int k = 0; k < kRuns; ++k)
                if (__shfl_sync(kFull, incl, own[k] + step - 1) <= base + 32 * k + lane) own[k] += step;
#pragma unroll
        for (int k = 0; k < kRuns; ++k) {
            const uint64_t o_rel = __shfl_sync(kFull, rel, own[k]);
            const uint32_t p = base + 32 * k + lane;
            u[k] = 0;
            if (p < total) u[k] = arena[o_rel + p];
        }
#pragma unroll
        for (int k = 0; k < kRuns; ++k)
            if (base + 32 * k + lane < total) f(own[k], u[k]);
    }
}

// Lanes adding to the same counter in one step (hub vertices recur across
// samples) are merged: one atomic per distinct address among the calling
// lanes, carrying the number of lanes.
__device__ __forceinline__ void add_aggregated(uint32_t* counter, int32_t u) {
    const unsigned active = __activemask();
    const unsigned peers = __match_any_sync(active, u);
    if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&counter[u], (uint32_t)__popc(peers));
}

// Greedy's cover walk: a block-local table merges the decrements of vertices
// that recur across the samples a seed covers (hubs), so that each such
// vertex takes one global atomic per block and round. A vertex that finds its
// slot held by another goes straight to the global counter.
constexpr int kHotBits = 10;
constexpr int kHotSlots = 1 << kHotBits;
constexpr uint32_t kHotEmpty = 0xFFFFFFFFu;

__device__ __forceinline__ void sub_merged(uint32_t* counter, int32_t u, uint32_t* hkey, uint32_t* hcnt) {
    const uint32_t slot = ((uint32_t)u * 2654435761u) >> (32 - kHotBits);
    uint32_t old = hkey[slot];
    if (old == kHotEmpty) old = atomicCAS(&hkey[slot], kHotEmpty, (uint32_t)u);
    if (old == kHotEmpty || old == (uint32_t)u) atomicAdd(&hcnt[slot], 1u);
    else atomicSub(&counter[u], 1u);
}

// ------------------------------------------------------------- coverage
// qbits (nullable): a filter of the batch's seeds, one bit per vertex for
// graphs of at most 2^20 vertices, else 2^20 bits indexed by a multiplicative
// hash, so that the sketch scan gathers a vertex's 8-byte mask only when the
// vertex may be a seed (false positives have an all-zero mask). At most
// 128 KiB: it fits in one block's shared memory.
constexpr int kFilterLog2 = 20;
constexpr uint32_t kFilterMaxWords = 1u << (kFilterLog2 - 5);

__host__ __device__ __forceinline__ uint32_t filter_words(int64_t n) {  // n in [1, 2^31]
    return n > ((int64_t)1 << kFilterLog2) ? kFilterMaxWords : (uint32_t)((n + 31) / 32);
}

__device__ __forceinline__ uint32_t filter_index(uint32_t v, int hashed) {
    return hashed ? (v * 2654435761u) >> (32 - kFilterLog2) : v;
}
__global__ void k_qmask_set(const int64_t* __restrict__ off, const int32_t* __restrict__ seeds, int32_t q0,
                            int32_t qn, int64_t n, uint64_t* __restrict__ qmask, uint32_t* __restrict__ qbits,
                            DevStatus* st, unsigned long long* __restrict__ reset3) {
    const int lane = threadIdx.x & 31;
    if (reset3 && blockIdx.x == 0 && threadIdx.x < 3) reset3[threadIdx.x] = 0;  // the ordered scan's counters
    const int32_t b = q0 + (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (b >= q0 + qn) return;
    const int64_t lo = off[b], hi = off[b + 1];
    const uint64_t bit = 1ull << (b - q0);
    if (hi <= lo && lane == 0) {
        atomicOr(&st->flags, kStInval);
        atomicMin(&st->first_bad, (unsigned long long)b);
    }
    for (int64_t i = lo + lane; i < hi; i += 32) {
        const int32_t v = seeds[i];
        bool bad = v < 0 || v >= n;
        if (!bad) bad = (atomicOr((unsigned long long*)&qmask[v], (unsigned long long)bit) & bit) != 0;
        if (!bad && qbits) {
            const uint32_t f = filter_index((uint32_t)v, n > ((int64_t)1 << kFilterLog2));
            atomicOr(&qbits[f >> 5], 1u << (f & 31));
        }
        if (bad) {
            atomicOr(&st->flags, kStInval);
            atomicMin(&st->first_bad, (unsigned long long)b);
        }
    }
}

// A warp takes 2^glog consecutive samples at a time. Bound by the chain of
// header, member and filter loads of the longest group: with 32 samples a warp
// a small sketch left most warp slots empty (ER 10k / 100k, 100K samples, 60
// members on average and up to 1,700: 3,125 groups for 9,728 slots, 76 us), so
// a group is only as large as keeps every slot supplied (coverage_shape), and
// four runs of 32 members are in flight. Without the bound on its registers the
// compiler takes 40, a quarter of the warp slots (64 queries of 679K samples of
// 70 members 182 us, 155 with 32).
__global__ void __launch_bounds__(kCovThreads, kCovBlocks) k_coverage(const uint64_t* __restrict__ h_off,
                                                          const uint32_t* __restrict__ h_len, uint64_t T,
                                                          const int32_t* __restrict__ arena,
                                                          const uint64_t* __restrict__ qmask,
                                                          const uint32_t* __restrict__ qbits, int hashed, int glog,
                                                          unsigned long long* __restrict__ cov) {
    __shared__ unsigned long long s_acc[kCovThreads / 32][32];
    __shared__ unsigned long long s_cnt[64];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    if (threadIdx.x < 64) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long c_lo = 0, c_hi = 0;  // counts of queries `lane` and `lane + 32`
    const uint64_t nwarps = (uint64_t)gridDim.x * (kCovThreads / 32);
    const uint64_t groups = (T + (1u << glog) - 1) >> glog;
    unsigned long long* acc_row = s_acc[wib];  // zero between groups
    acc_row[lane] = 0;
    __syncwarp();
    for (uint64_t gidx = (uint64_t)blockIdx.x * (kCovThreads / 32) + wib; gidx < groups; gidx += nwarps) {
        const uint64_t j = (gidx << glog) + lane;
        const bool valid = lane < (1 << glog) && j < T;
        const uint64_t off = valid ? h_off[j] : 0;
        const uint32_t len = valid ? h_len[j] : 0;
        bool hit = false;
        warp_members<4>(off, len, arena, [&](int owner, int32_t u) {
            if (qbits) {  // not a seed
                const uint32_t f = filter_index((uint32_t)u, hashed);
                if (!((__ldg(qbits + (f >> 5)) >> (f & 31)) & 1u)) return;
            }
            const uint64_t msk = qmask[u];
            if (msk) {
                atomicOr(&acc_row[owner], (unsigned long long)msk);
                hit = true;
            }
        });
        if (!__any_sync(kFull, hit)) continue;
        __syncwarp();  // every lane has the others' ORs (a vote orders no memory)
        const uint64_t acc = acc_row[lane];
        acc_row[lane] = 0;
        __syncwarp();
        uint64_t present = (uint64_t)__reduce_or_sync(kFull, (uint32_t)(acc >> 32)) << 32 |
                           __reduce_or_sync(kFull, (uint32_t)acc);
        while (present) {
            const int b = __ffsll((long long)present) - 1;
            present &= present - 1;
            const unsigned c = (unsigned)__popc(__ballot_sync(kFull, (acc >> b) & 1ull));
            if (lane == (b & 31)) {
                if (b < 32) c_lo += c;
                else c_hi += c;
            }
        }
    }
    if (c_lo) atomicAdd(&s_cnt[lane], c_lo);
    if (c_hi) atomicAdd(&s_cnt[lane + 32], c_hi);
    __syncthreads();
    if (threadIdx.x < 64 && s_cnt[threadIdx.x]) atomicAdd(&cov[threadIdx.x], s_cnt[threadIdx.x]);
}

// The scan of a sketch whose members are in sample-id order (arena
// positions [h_off[0], ...) contiguous): the seed filter sits in shared
// memory; a warp takes a task of 2^tlog consecutive samples at a time (from an
// atomic cursor, so that warps meeting many seeds take fewer), whose members
// are one run, and streams it as 16-byte vectors testing each member against
// the filter. Possible seeds (rare) are held back per warp and join the hit
// list for k_scan_hits with one atomic for dozens; only when the list is full
// is a hit resolved here. The first setter of a (sample, query) bit of smask
// counts it, and the first setter of a sample's word lists the sample for the
// reset. Bound by the returning list atomics when each hit took one on the same
// counter, and by too few tasks where samples are large (1024 samples a task):
// 10M samples of 4 members and 64 queries of 10 seeds 71 -> 53 us, the whole
// call 177 -> 168; 1M of 70 members 309 -> 175; 6M of 4 members and 64 queries
// of 250 seeds 778 -> 470. Now by the chain of load, filter read and branch at
// one block an SM (the filter's 128 KiB); the members' bytes alone take 25 us.
constexpr int kScanThreads = 1024;

// Asynchronous bulk prefetch of [p, p + bytes) into L2 (p 16-byte aligned,
// bytes a multiple of 16): no register waits for it.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
constexpr int kScanUnroll = 4;
constexpr unsigned int kScanHits = 128;  // hits a warp holds back
constexpr uint64_t kScanMembers = 2048;
constexpr uint64_t kScanAhead = 8;  // warp steps prefetched ahead
constexpr unsigned long long kHitCap = 1ull << 22;  // hits listed per query chunk (32 MiB); more are resolved in the scan

__global__ void __launch_bounds__(kScanThreads, 1) k_scan_ordered(
    const uint64_t* __restrict__ h_off, const uint32_t* __restrict__ h_len, uint64_t T, int tlog,
    const int32_t* __restrict__ arena, const uint32_t* __restrict__ qbits, uint32_t fwords, int hashed,
    const uint64_t* __restrict__ qmask, unsigned long long* __restrict__ smask, uint32_t* __restrict__ touched,
    unsigned long long* __restrict__ ntouched, unsigned long long* __restrict__ cursor,
    unsigned long long* __restrict__ hits, unsigned long long* __restrict__ nhits, unsigned long long hit_cap,
    unsigned long long* __restrict__ cov) {
    extern __shared__ __align__(16) uint32_t s_f[];
    __shared__ unsigned int s_cnt[64];
    __shared__ unsigned long long s_hit[kScanThreads / 32][kScanHits];
    __shared__ unsigned int s_nhit[kScanThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint4* q4 = reinterpret_cast<const uint4*>(qbits);
#pragma unroll 8
    for (uint32_t i = threadIdx.x; i < fwords / 4; i += kScanThreads) reinterpret_cast<uint4*>(s_f)[i] = q4[i];
    if (threadIdx.x < fwords % 4) s_f[(fwords & ~3u) + threadIdx.x] = qbits[(fwords & ~3u) + threadIdx.x];
    if (threadIdx.x < 64) s_cnt[threadIdx.x] = 0;
    if (lane == 0) s_nhit[wid] = 0;
    __syncthreads();
    unsigned long long* const my_hit = s_hit[wid];
    // hit h = (task << 40) | position takes place `slot` of the list; where that
    // is full, it is resolved here: the member's query mask, its sample (the
    // last whose run starts at or before it) and the counts
    auto list = [&](unsigned long long h, unsigned long long slot) {
        if (slot < hit_cap) {
            hits[slot] = h;
            return;
        }
        const uint64_t pos = h & ((1ull << 40) - 1);
        const uint64_t msk = qmask[arena[pos]];
        if (!msk) return;  // a filter collision
        uint64_t lo = (h >> 40) << tlog, hi = min(T, lo + (1u << tlog)) - 1;
        while (lo < hi) {
            const uint64_t mid = (lo + hi + 1) >> 1;
            if (h_off[mid] <= pos) lo = mid;
            else hi = mid - 1;
        }
        const unsigned long long old = atomicOr(smask + lo, (unsigned long long)msk);
        if (old == 0) touched[atomicAdd(ntouched, 1ull)] = (uint32_t)lo;
        for (uint64_t nb = msk & ~old; nb; nb &= nb - 1) atomicAdd(&s_cnt[__ffsll((long long)nb) - 1], 1u);
    };
    // the warp's hits join the list, one atomic for all
    auto flush = [&](unsigned int cnt) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(nhits, (unsigned long long)cnt);
        base = __shfl_sync(kFull, base, 0);
        for (unsigned int i = lane; i < cnt; i += 32) list(my_hit[i], base + i);
        __syncwarp();
        if (lane == 0) s_nhit[wid] = 0;
        __syncwarp();
    };
    const uint64_t ntask = (T + (1u << tlog) - 1) >> tlog;
    unsigned long long claim = 0;
    if (lane == 0) claim = atomicAdd(cursor, 1ull);
    for (;;) {
        const unsigned long long task = __shfl_sync(kFull, claim, 0);
        if (task >= ntask) break;
        if (lane == 0) claim = atomicAdd(cursor, 1ull);  // the next task, claimed while this one streams
        const uint64_t j0 = task << tlog, j1 = min(T, j0 + (1u << tlog));
        const uint64_t p0 = h_off[j0], p1 = h_off[j1 - 1] + h_len[j1 - 1];
        auto member = [&](uint64_t pos, int32_t u) {
            const uint32_t f = filter_index((uint32_t)u, hashed);
            if (!((s_f[f >> 5] >> (f & 31)) & 1u)) return;
            // a possible seed: its (task, position) goes to the hit list for k_scan_hits
            const unsigned int slot = atomicAdd(&s_nhit[wid], 1u);
            if (slot < kScanHits) my_hit[slot] = ((unsigned long long)task << 40) | pos;
            else list(((unsigned long long)task << 40) | pos, atomicAdd(nhits, 1ull));
        };
        const uint64_t up = (p0 + 3) & ~(uint64_t)3, down = p1 & ~(uint64_t)3;
        const uint64_t ph = p1 < up ? p1 : up, pt = down > ph ? down : ph;
        if (p0 + lane < ph) member(p0 + lane, arena[p0 + lane]);
        const int4* a4 = reinterpret_cast<const int4*>(arena);
        const uint64_t v_end = pt / 4, v0 = ph / 4;
        // the task's first steps, then each step the one kScanAhead steps on, are
        // prefetched into L2 by one lane, so that the lanes' loads find them there
        constexpr uint64_t kStep = 32 * kScanUnroll;  // 16-byte vectors a warp step loads
        if (lane == 0 && v0 < v_end)
            prefetch_l2(a4 + v0, (uint32_t)(min(v_end - v0, kStep * kScanAhead) * 16));
        // kScanUnroll 16-byte loads in flight a lane before any member is tested
        // (the last step of a task predicated, not a step per load)
        for (uint64_t vb = v0; vb < v_end; vb += kStep) {
            const uint64_t ahead = vb + kStep * kScanAhead, v = vb + lane;
            if (lane == 0 && ahead < v_end) prefetch_l2(a4 + ahead, (uint32_t)(min(v_end - ahead, kStep) * 16));
            int4 m[kScanUnroll];
#pragma unroll
            for (int k = 0; k < kScanUnroll; ++k)
                if (v + 32 * k < v_end) m[k] = __ldcs(a4 + v + 32 * k);
#pragma unroll
            for (int k = 0; k < kScanUnroll; ++k) {
                if (v + 32 * k >= v_end) break;
                const uint64_t pos = (v + 32 * k) * 4;
                member(pos, m[k].x);
                member(pos + 1, m[k].y);
                member(pos + 2, m[k].z);
                member(pos + 3, m[k].w);
            }
            __syncwarp();
            // one lane's read decides for the warp (a lane of its own might already see the next step's hits)
            const unsigned int cnt = __shfl_sync(kFull, s_nhit[wid], 0);
            if (cnt >= kScanHits / 2) flush(min(cnt, kScanHits));
        }
        if (pt + lane < p1) member(pt + lane, arena[pt + lane]);
    }
    __syncwarp();
    const unsigned int rest = __shfl_sync(kFull, s_nhit[wid], 0);
    if (rest) flush(min(rest, kScanHits));
    __syncthreads();
    if (threadIdx.x < 64 && s_cnt[threadIdx.x]) atomicAdd(&cov[threadIdx.x], (unsigned long long)s_cnt[threadIdx.x]);
}

// Samples of a scan task, as a power of two: about kScanMembers members (of
// 1024, 2048, 4096 members a task the calls above took 183, 168, 178 us, 185,
// 179, 190 and 470, 469, 520), and the tasks' numbers fit the 24 bits of a hit.
static int scan_task_log(uint64_t T, uint64_t members) {
    int tlog = 5;
    while (tlog < 10 && (members << tlog) < kScanMembers * T) ++tlog;
    while ((T >> tlog) >= (1ull << 24) - 1) ++tlog;
    return tlog;
}

// The hits the scan listed: each (task, position) resolves to its member,
// the member's query mask, and its sample by a binary search over the task's
// offsets; the first setter of a (sample, query) bit counts it.
__global__ void __launch_bounds__(256) k_scan_hits(const unsigned long long* __restrict__ hits,
                                                   const unsigned long long* __restrict__ nhits,
                                                   unsigned long long hit_cap, const uint64_t* __restrict__ h_off,
                                                   uint64_t T, int tlog, const int32_t* __restrict__ arena,
                                                   const uint64_t* __restrict__ qmask,
                                                   unsigned long long* __restrict__ smask,
                                                   uint32_t* __restrict__ touched,
                                                   unsigned long long* __restrict__ ntouched,
                                                   unsigned long long* __restrict__ cov) {
    __shared__ unsigned int s_cnt[64];
    if (threadIdx.x < 64) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t cnt = min((uint64_t)*nhits, (uint64_t)hit_cap);
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < cnt; k += (uint64_t)gridDim.x * blockDim.x) {
        const unsigned long long h = hits[k];
        const uint64_t pos = h & ((1ull << 40) - 1), task = h >> 40;
        const uint64_t msk = qmask[arena[pos]];
        if (!msk) continue;  // a filter collision
        uint64_t lo = task << tlog, hi = min(T, lo + (1u << tlog)) - 1;
        while (lo < hi) {
            const uint64_t mid = (lo + hi + 1) >> 1;
            if (h_off[mid] <= pos) lo = mid;
            else hi = mid - 1;
        }
        const unsigned long long old = atomicOr(smask + lo, (unsigned long long)msk);
        if (old == 0) touched[atomicAdd(ntouched, 1ull)] = (uint32_t)lo;
        for (uint64_t nb = msk & ~old; nb; nb &= nb - 1) atomicAdd(&s_cnt[__ffsll((long long)nb) - 1], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 64 && s_cnt[threadIdx.x]) atomicAdd(&cov[threadIdx.x], (unsigned long long)s_cnt[threadIdx.x]);
}

// Eq. 21 with exact integers: N = Cov W + T sum_{v in S} (2^f - w_v),
// D = T 2^f, estimate = N / D, of query b by one warp (Cov = c).
__device__ __forceinline__ void estimate_query(const int64_t* __restrict__ off, const int32_t* __restrict__ seeds,
                                               int32_t b, int64_t n, const uint64_t* __restrict__ w, int f, uint64_t W,
                                               uint64_t T, uint64_t c, int64_t* __restrict__ cov_out,
                                               double* __restrict__ est_out, int ris) {
    const int lane = threadIdx.x & 31;
    const uint64_t one_f = 1ull << f;
    uint64_t s = 0;  // <= |S| 2^f <= 2^61
    for (int64_t i = off[b] + lane; i < off[b + 1]; i += 32) {
        const int32_t v = seeds[i];
        if (v >= 0 && v < n) s += one_f - w[v];
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(kFull, s, d);
    if (lane == 0) {
        // RIS (Lemma 1): n Cov / T; SKIS (Eq. 21): (Cov W + T sum) / (T 2^f)
        const u128 N = ris ? (u128)c * (uint64_t)n : (u128)c * W + (u128)T * s;
        const u128 D = ris ? (u128)T : (u128)T << f;
        if (cov_out) cov_out[b] = (int64_t)c;
        est_out[b] = u128_to_double(N) / u128_to_double(D);
    }
}

__global__ void k_estimate(const int64_t* __restrict__ off, const int32_t* __restrict__ seeds, int32_t q0,
                           int32_t qn, int64_t n, const uint64_t* __restrict__ w, int f, uint64_t W, uint64_t T,
                           const unsigned long long* __restrict__ cov, int64_t* __restrict__ cov_out,
                           double* __restrict__ est_out, int ris) {
    const int32_t b = q0 + (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (b >= q0 + qn) return;
    estimate_query(off, seeds, b, n, w, f, W, T, cov[b - q0], cov_out, est_out, ris);
}

// The end of a batch of queries, a warp each: the estimate, and everything the
// batch set goes back to zero (its seeds' masks and filter bits, its coverage
// counts and, by the blocks past the queries', the samples' query words).
// status_out (nullable) receives the status word.
__global__ void k_finish(const int64_t* __restrict__ off, const int32_t* __restrict__ seeds, int32_t q0, int32_t qn,
                         int64_t n, const uint64_t* __restrict__ w, int f, uint64_t W, uint64_t T,
                         unsigned long long* __restrict__ cov, int64_t* __restrict__ cov_out,
                         double* __restrict__ est_out, int ris, uint64_t* __restrict__ qmask,
                         uint32_t* __restrict__ qbits, int qblocks, const uint32_t* __restrict__ touched,
                         const unsigned long long* __restrict__ ntouched, unsigned long long* __restrict__ smask,
                         const DevStatus* __restrict__ status, DevStatus* __restrict__ status_out) {
    if ((int)blockIdx.x >= qblocks) {
        const uint64_t cnt = *ntouched;
        for (uint64_t k = (uint64_t)(blockIdx.x - qblocks) * blockDim.x + threadIdx.x; k < cnt;
             k += (uint64_t)(gridDim.x - qblocks) * blockDim.x)
            smask[touched[k]] = 0;
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (status_out) *status_out = *status;
        cov[64] = 0;  // the index walk's queue
    }
    const int lane = threadIdx.x & 31;
    const int32_t b = q0 + (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (b >= q0 + qn) return;
    const uint64_t c = cov[b - q0];
    estimate_query(off, seeds, b, n, w, f, W, T, c, cov_out, est_out, ris);
    if (lane == 0) cov[b - q0] = 0;
    for (int64_t i = off[b] + lane; i < off[b + 1]; i += 32) {
        const int32_t v = seeds[i];
        if (v >= 0 && v < n) {
            qmask[v] = 0;
            // every bit set in the filter belongs to a seed of this batch
            if (qbits) qbits[filter_index((uint32_t)v, n > ((int64_t)1 << kFilterLog2)) >> 5] = 0;
        }
    }
}

#define CV_CUDA(call)                                                              \
    do {                                                                           \
        cudaError_t _e = (call);                                                   \
        if (_e != cudaSuccess) {                                                   \
            *err = std::string(where) + ": CUDA error: " + cudaGetErrorString(_e); \
            return _e == cudaErrorMemoryAllocation ? SKIS_ENOMEM : SKIS_ERR_CUDA;  \
        }                                                                          \
    } while (0)

static int coverage_blocks(uint64_t T) {
    const uint64_t groups = (T + 31) / 32;
    const uint64_t want = (groups + (kCovThreads / 32) - 1) / (kCovThreads / 32);
    return (int)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)sm_count() * 8));
}

// k_coverage's grid and group size: the largest groups (at most 32 samples)
// that still give two to each of the GPU's warps.
void coverage_shape(uint64_t T, int* blocks, int* glog) {
    const uint64_t warps = (uint64_t)sm_count() * kCovBlocks * (kCovThreads / 32);
    *glog = 5;
    while (*glog > 0 && (T >> *glog) < 2 * warps) --*glog;
    const uint64_t groups = (T + (1u << *glog) - 1) >> *glog;
    const uint64_t want = (groups + kCovThreads / 32 - 1) / (kCovThreads / 32);
    *blocks = (int)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)sm_count() * kCovBlocks));
}

// ------------------------------------------- coverage by inverted index
// Cov_R(S) for small seed sets: walk the sample list of every seed and set
// the query's bit in a per-sample mask; the first setter of (sample, query)
// counts it. A warp takes a seed and the first kInvChunk entries of its list;
// the further chunks of a long list (a hub's) are queued and dealt over the
// grid by the next launch, or, past the queue's capacity, walked on the spot.
// Bound by latency: seed, list bounds, list and mask are one dependent load
// after another, so the lists are short work in many warps, four entries a
// lane in flight. 64 queries, 13,800 seeds, lists of 93 entries on average
// (Chung-Lu 4M / 70M WC, 5M samples): set and reset 117 us with a chunk table,
// its prefix sums and a search of it per chunk of 2048, in seven launches; 154,
// 66 and 50 us like this with chunks of 2048, 512 and 256.
constexpr uint32_t kInvChunk = 256;
// queue item: the seed's place in the batch (below 64 n <= 2^37) and the chunk
// of its list (below 2^32 / kInvChunk = 2^24: a list holds a sample once)
constexpr int kInvChunkBits = 24;

struct InvWalk {
    const int64_t* off;     // the batch's seed offsets and seeds
    const int32_t* seeds;
    int32_t q0, qn;
    int64_t seed_base, nseeds, n;
    const uint64_t* inv_off;
    const uint32_t* inv;
    unsigned long long* smask;
    unsigned long long* cov;      // qn counts
    uint64_t* queue;              // seed << kInvChunkBits | chunk
    uint64_t queue_cap;
    unsigned long long* nqueue;   // chunks queued or past the capacity
};

// Sets `bit` in the masks of list entries [x0, x1) (clear: zeroes the masks);
// returns how many masks of the lane's entries did not have it.
__device__ __forceinline__ uint32_t walk_list(const InvWalk& a, uint64_t x0, uint64_t x1, unsigned long long bit, bool clear) {
    uint32_t fresh = 0;
    for (uint64_t x = x0 + (threadIdx.x & 31); x < x1; x += 128) {
        uint32_t j[4];
        unsigned long long old[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (x + 32 * q < x1) j[q] = a.inv[x + 32 * q];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            old[q] = bit;
            if (x + 32 * q < x1) {
                if (clear) a.smask[j[q]] = 0;
                else old[q] = atomicOr(&a.smask[j[q]], bit);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) fresh += (old[q] & bit) ? 0u : 1u;
    }
    return fresh;
}

// mode 0: the lists' first chunks (the others queued); 1: the queued chunks;
// 2: every mask they set back to zero
__global__ void __launch_bounds__(kCovThreads) k_cover_inv(InvWalk a, int mode) {
    __shared__ int64_t s_off[65];
    __shared__ unsigned int s_cov[64];
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i <= a.qn; i += kCovThreads) s_off[i] = a.off[a.q0 + i];
    if (threadIdx.x < 64) s_cov[threadIdx.x] = 0;
    __syncthreads();
    auto query_of = [&](int64_t i) -> int {  // the last query b with off[b] <= seed_base + i
        int lo = 0, hi = a.qn - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (s_off[mid] <= a.seed_base + i) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    auto add = [&](int b, uint32_t fresh) {
        fresh = __reduce_add_sync(kFull, fresh);
        if (lane == 0 && fresh) atomicAdd(&s_cov[b], fresh);
    };
    const int64_t nwarps = (int64_t)gridDim.x * (kCovThreads / 32);
    const int64_t w0 = ((int64_t)blockIdx.x * kCovThreads + threadIdx.x) / 32;
    const uint64_t queued = mode ? min((uint64_t)*a.nqueue, a.queue_cap) : 0;
    const bool past = mode == 2 && *a.nqueue > a.queue_cap;
    if (mode != 1) {
        for (int64_t i = w0; i < a.nseeds; i += nwarps) {
            const int32_t v = a.seeds[a.seed_base + i];
            if (v < 0 || v >= a.n) continue;
            const uint64_t lo = a.inv_off[v], len = a.inv_off[v + 1] - lo;
            const int b = query_of(i);
            const unsigned long long bit = 1ull << b;
            uint64_t rest = len;  // entries [rest, len) are walked here as well
            if (len > kInvChunk) {
                if (mode == 2) {
                    if (past) rest = kInvChunk;  // whichever were queued, all of it
                } else {
                    const uint64_t more = (len - 1) / kInvChunk;
                    unsigned long long at = 0;
                    if (lane == 0) at = atomicAdd(a.nqueue, (unsigned long long)more);
                    at = __shfl_sync(kFull, at, 0);
                    const uint64_t fit = at < a.queue_cap ? min(more, (uint64_t)(a.queue_cap - at)) : 0;
                    for (uint64_t c = lane; c < fit; c += 32) a.queue[at + c] = ((uint64_t)i << kInvChunkBits) | (c + 1);
                    rest = min(len, (fit + 1) * kInvChunk);
                }
            }
            uint32_t fresh = walk_list(a, lo, lo + min(len, (uint64_t)kInvChunk), bit, mode == 2);
            if (rest < len) fresh += walk_list(a, lo + rest, lo + len, bit, mode == 2);
            if (mode == 0) add(b, fresh);
        }
    }
    for (uint64_t k = w0; k < queued; k += nwarps) {
        const uint64_t item = a.queue[k];
        const int64_t i = (int64_t)(item >> kInvChunkBits);
        const int32_t v = a.seeds[a.seed_base + i];
        const uint64_t x = a.inv_off[v] + (item & ((1u << kInvChunkBits) - 1u)) * kInvChunk;
        const int b = query_of(i);
        const uint32_t fresh = walk_list(a, x, min(x + kInvChunk, a.inv_off[v + 1]), 1ull << b, mode == 2);
        if (mode == 1) add(b, fresh);
    }
    if (mode == 2) return;
    __syncthreads();
    if (threadIdx.x < 64 && s_cov[threadIdx.x]) atomicAdd(&a.cov[threadIdx.x], (unsigned long long)s_cov[threadIdx.x]);
}

cudaError_t coverage_by_index(const skis_sketch* s, const int64_t* off, const int32_t* seeds, int32_t q0,
                              int32_t qn, int64_t seed_base, int64_t nseeds, uint64_t* queue, uint64_t queue_cap,
                              uint64_t* smask, unsigned long long* cov, cudaStream_t st) {
    if (nseeds <= 0) return cudaSuccess;
    InvWalk a;
    a.off = off;
    a.seeds = seeds;
    a.q0 = q0;
    a.qn = qn;
    a.seed_base = seed_base;
    a.nseeds = nseeds;
    a.n = s->g->n;
    a.inv_off = s->inv_off;
    a.inv = s->inv;
    a.smask = reinterpret_cast<unsigned long long*>(smask);
    a.cov = cov;
    a.queue = queue;
    a.queue_cap = queue_cap;
    a.nqueue = cov + 64;
    const int full = sm_count() * 8;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((nseeds + kCovThreads / 32 - 1) / (kCovThreads / 32), full));
    k_cover_inv<<<blocks, kCovThreads, 0, st>>>(a, 0); note_launch();
    k_cover_inv<<<full, kCovThreads, 0, st>>>(a, 1); note_launch();
    k_cover_inv<<<full, kCovThreads, 0, st>>>(a, 2); note_launch();
    return cudaGetLastError();
}

// Members of samples [0, cnt) (headers off/len) copied to out in sample
// order at their exclusive prefix pre: a warp takes 32 consecutive samples
// and spreads their members over its lanes, so the writes are one
// contiguous run.
__global__ void __launch_bounds__(kCovThreads) k_order_members(const uint64_t* __restrict__ off,
                                                               const uint32_t* __restrict__ len, uint64_t cnt,
                                                               const uint64_t* __restrict__ pre,
                                                               const int32_t* __restrict__ arena,
                                                               int32_t* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const uint64_t nwarps = (uint64_t)gridDim.x * (kCovThreads / 32);
    for (uint64_t gi = ((uint64_t)blockIdx.x * kCovThreads + threadIdx.x) / 32; gi * 32 < cnt; gi += nwarps) {
        const uint64_t j = gi * 32 + lane;
        const uint64_t o = j < cnt ? off[j] : 0;
        const uint32_t l = j < cnt ? len[j] : 0u;
        uint32_t incl = l;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += y;
        }
        const uint32_t total = __shfl_sync(kFull, incl, 31), excl = incl - l;
        const uint64_t dst0 = pre[gi * 32];
        for (uint32_t base = 0; base < total; base += 32) {  // warp-uniform: every lane shuffles
            const uint32_t p = base + lane;
            int owner = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const uint32_t v = __shfl_sync(kFull, incl, owner + step - 1);
                if (v <= p) owner += step;
            }
            const uint64_t oo = __shfl_sync(kFull, o, owner);
            const uint32_t oe = __shfl_sync(kFull, excl, owner);
            if (p < total) out[dst0 + p] = arena[oo + (p - oe)];
        }
    }
}

__global__ void k_rebase_offsets(uint64_t* __restrict__ off, const uint64_t* __restrict__ pre, uint64_t cnt,
                                 uint64_t base) {
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < cnt; j += (uint64_t)gridDim.x * blockDim.x)
        off[j] = base + pre[j];
}

int sketch_order_arena(skis_sketch* s, cudaStream_t st, std::string* err) {
    const char* where = "member layout";
    if (s->ordered_T == s->T) return SKIS_OK;
    const uint64_t T0 = s->ordered_T, cnt = s->T - T0, E0 = s->ordered_E;
    uint64_t* pre = nullptr;
    int32_t* tmp = nullptr;
    uint64_t E1 = 0;
    auto body = [&]() -> int {
        CV_CUDA(dev_alloc_t(&pre, (size_t)cnt + 1, st));
        CV_CUDA(scan_u32_to_u64(s->h_len + T0, pre, (int64_t)cnt, st));
        CV_CUDA(cudaMemcpyAsync(&E1, pre + cnt, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
        CV_CUDA(cudaStreamSynchronize(st));
        CV_CUDA(dev_alloc_t(&tmp, (size_t)std::max<uint64_t>(E1, 1), st));
        const int blocks = (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)sm_count() * 8,
                                                                         (cnt + kCovThreads - 1) / kCovThreads));
        k_order_members<<<blocks, kCovThreads, 0, st>>>(s->h_off + T0, s->h_len + T0, cnt, pre, s->arena, tmp);
        note_launch();
        CV_CUDA(cudaGetLastError());
        if (E1) CV_CUDA(cudaMemcpyAsync(s->arena + E0, tmp, E1 * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
        k_rebase_offsets<<<blocks, kCovThreads, 0, st>>>(s->h_off + T0, pre, cnt, E0); note_launch();
        CV_CUDA(cudaGetLastError());
        if (s->ctr) {  // later samples are appended right after the ordered ones
            const unsigned long long cur = E0 + E1;
            CV_CUDA(cudaMemcpyAsync(&s->ctr->arena, &cur, sizeof(cur), cudaMemcpyHostToDevice, st));
        }
        s->arena_used = E0 + E1;
        s->arena_drawn = s->T;
        s->arena_ends = 0;
        CV_CUDA(cudaStreamSynchronize(st));
        return SKIS_OK;
    };
    const int rc = body();
    dev_free(pre, st);
    dev_free(tmp, st);
    if (rc == SKIS_OK) {
        s->ordered_T = s->T;
        s->ordered_E = E0 + E1;
    }
    return rc;
}

static int estimate_queries(skis_sketch* s, int32_t q, const int64_t* d_off, const int32_t* d_seeds,
                            const int64_t* h_off, int64_t* d_cov, double* d_est, cudaStream_t st, std::string* err,
                            void* d_pack, void* h_pack, size_t pack_bytes) {
    const char* where = "skis_estimate";
    const skis_graph* g = s->g;
    if (s->T == 0) {
        *err = "skis_estimate: the sketch has no samples";
        return SKIS_EINVAL;
    }
    if (s->query_index == 1) {
        const int rc = sketch_inverted(s, st, err);
        if (rc != SKIS_OK) return rc;
    }
    const bool by_index = s->query_index < 2 && s->inv && s->inv_T == s->T;
    // a large sketch is scanned with its members in sample-id order (laid out
    // once per new samples); a small one (below 2^20 samples: doubling rounds,
    // tests) directly, where that one-time layout would cost more than it saves
    const bool ordered_scan = !by_index && (s->T >= (1ull << 20) || s->query_index == 3) && s->T < (1ull << 32);
    if (ordered_scan) {
        const int rc = sketch_order_arena(s, st, err);
        if (rc != SKIS_OK) return rc;
    }
    const uint32_t fwords = filter_words(g->n);
    const int hashed = g->n > ((int64_t)1 << kFilterLog2);
    // each buffer by its own pointer: a call that ran out of memory may have left any of them
    if (!s->qmask) {
        CV_CUDA(dev_alloc_t(&s->qmask, (size_t)g->n, st));
        CV_CUDA(cudaMemsetAsync(s->qmask, 0, (size_t)g->n * sizeof(uint64_t), st));
    }
    if (!s->qbits) {
        CV_CUDA(dev_alloc_t(&s->qbits, (size_t)fwords, st));
        CV_CUDA(cudaMemsetAsync(s->qbits, 0, (size_t)fwords * sizeof(uint32_t), st));
    }
    // coverage counts, the index walk's queue length and the status, zero
    // (first_bad all ones) between calls
    if (!s->qcov) {
        CV_CUDA(dev_alloc_t(&s->qcov, 65, st));
        CV_CUDA(cudaMemsetAsync(s->qcov, 0, 65 * sizeof(unsigned long long), st));
    }
    if (!s->qstatus) {
        CV_CUDA(dev_alloc_t(&s->qstatus, 1, st));
        CV_CUDA(cudaMemsetAsync(s->qstatus, 0, sizeof(DevStatus), st));
        CV_CUDA(cudaMemsetAsync(&s->qstatus->first_bad, 0xFF, sizeof(unsigned long long), st));
    }
    for (int i = 0; i < 2; ++i)
        if (!s->qev[i]) CV_CUDA(cudaEventCreate(&s->qev[i]));
    uint64_t* queue = nullptr;
    uint64_t queue_cap = 0;
    if (ordered_scan) {
        if (s->touched_cap < s->T) {
            s->touched_cap = 0;
            dev_free(s->touched, st);
            s->touched = nullptr;
            CV_CUDA(dev_alloc_t(&s->touched, (size_t)s->T, st));
            s->touched_cap = s->T;
        }
        // list count, task cursor and hit count (k_qmask_set resets them)
        if (!s->ntouched) CV_CUDA(dev_alloc_t(&s->ntouched, 3, st));
        if (!s->hits) CV_CUDA(dev_alloc_t(&s->hits, (size_t)kHitCap, st));
    }
    if (by_index || ordered_scan) {
        if (s->smask_cap < s->T) {
            s->smask_cap = 0;
            dev_free(s->smask, st);
            s->smask = nullptr;
            CV_CUDA(dev_alloc_t(&s->smask, (size_t)s->T, st));
            CV_CUDA(cudaMemsetAsync(s->smask, 0, (size_t)s->T * sizeof(uint64_t), st));
            s->smask_cap = s->T;
        }
    }
    if (by_index) {
        int64_t most = 1;
        for (int32_t q0 = 0; q0 < q; q0 += 64)
            most = std::max<int64_t>(most, h_off[std::min<int32_t>(q, q0 + 64)] - h_off[q0]);
        queue_cap = (uint64_t)most + kInvQueueExtra;
        CV_CUDA(dev_alloc_t(&queue, (size_t)queue_cap, st));
    }
    if (ordered_scan)  // the filter takes up to 128 KiB of dynamic shared memory
        CV_CUDA(cudaFuncSetAttribute(k_scan_ordered, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(kFilterMaxWords * sizeof(uint32_t))));
    int cblocks = 0, glog = 0;
    coverage_shape(s->T, &cblocks, &glog);
    const int tlog = scan_task_log(s->T, s->arena_used);
    float query_ms = 0;
    for (int32_t q0 = 0; q0 < q; q0 += 64) {
        const int32_t qn = std::min<int32_t>(64, q - q0);
        const int wb = div_up((int64_t)qn * 32, 256);
        k_qmask_set<<<wb, 256, 0, st>>>(d_off, d_seeds, q0, qn, g->n, s->qmask, s->qbits, s->qstatus,
                                        ordered_scan ? s->ntouched : nullptr); note_launch();
        CV_CUDA(cudaGetLastError());
        CV_CUDA(cudaEventRecord(s->qev[0], st));
        if (by_index) {
            CV_CUDA(coverage_by_index(s, d_off, d_seeds, q0, qn, h_off[q0], h_off[q0 + qn] - h_off[q0], queue,
                                      queue_cap, s->smask, s->qcov, st));
        } else if (ordered_scan) {
            k_scan_ordered<<<sm_count(), kScanThreads, fwords * sizeof(uint32_t), st>>>(
                s->h_off, s->h_len, s->T, tlog, s->arena, s->qbits, fwords, hashed, s->qmask,
                reinterpret_cast<unsigned long long*>(s->smask), s->touched, s->ntouched, s->ntouched + 1, s->hits,
                s->ntouched + 2, kHitCap, s->qcov);
            note_launch();
            CV_CUDA(cudaGetLastError());
            k_scan_hits<<<sm_count() * 8, 256, 0, st>>>(s->hits, s->ntouched + 2, kHitCap, s->h_off, s->T, tlog, s->arena,
                                                        s->qmask, reinterpret_cast<unsigned long long*>(s->smask),
                                                        s->touched, s->ntouched, s->qcov);
            note_launch();
            CV_CUDA(cudaGetLastError());
        } else {
            k_coverage<<<cblocks, kCovThreads, 0, st>>>(s->h_off, s->h_len, s->T, s->arena, s->qmask, s->qbits, hashed,
                                                        glog, s->qcov);
            note_launch();
            CV_CUDA(cudaGetLastError());
        }
        CV_CUDA(cudaEventRecord(s->qev[1], st));
        k_finish<<<wb + (ordered_scan ? sm_count() : 0), 256, 0, st>>>(
            d_off, d_seeds, q0, qn, g->n, g->w, g->f, g->W, s->T, s->qcov, d_cov, d_est, s->ris, s->qmask, s->qbits, wb,
            s->touched, s->ntouched, reinterpret_cast<unsigned long long*>(s->smask), s->qstatus,
            static_cast<DevStatus*>(d_pack));
        note_launch();
        CV_CUDA(cudaGetLastError());
    }
    dev_free(queue, st);
    DevStatus h;
    if (d_pack) CV_CUDA(cudaMemcpyAsync(h_pack, d_pack, pack_bytes, cudaMemcpyDeviceToHost, st));
    else CV_CUDA(cudaMemcpyAsync(&h, s->qstatus, sizeof(DevStatus), cudaMemcpyDeviceToHost, st));
    CV_CUDA(cudaStreamSynchronize(st));
    if (d_pack) h = *static_cast<const DevStatus*>(h_pack);
    if (q > 0 && q <= 64) {  // the device time of the coverage launches (one chunk of queries)
        cudaEventElapsedTime(&query_ms, s->qev[0], s->qev[1]);
        s->last_query_ms = query_ms;
    }
    if (h.flags & kStInval) {
        CV_CUDA(cudaMemsetAsync(s->qstatus, 0, sizeof(DevStatus), st));
        CV_CUDA(cudaMemsetAsync(&s->qstatus->first_bad, 0xFF, sizeof(unsigned long long), st));
        *err = "skis_estimate: query " + std::to_string(h.first_bad) +
               " is empty, has a seed outside [0, n) or repeats a seed";
        return SKIS_EINVAL;
    }
    return SKIS_OK;
}

int sketch_estimate(skis_sketch* s, int32_t q, const int64_t* d_off, const int32_t* d_seeds, const int64_t* h_off,
                    int64_t* d_cov, double* d_est, cudaStream_t st, std::string* err, void* d_pack, void* h_pack,
                    size_t pack_bytes) {
    return with_room(s, st, err, [&] {  // every buffer is there before the first launch
        return estimate_queries(s, q, d_off, d_seeds, h_off, d_cov, d_est, st, err, d_pack, h_pack, pack_bytes);
    });
}

// --------------------------------------------------------------- greedy
__global__ void __launch_bounds__(kCovThreads) k_count_members(const uint64_t* __restrict__ h_off,
                                                               const uint32_t* __restrict__ h_len, uint64_t T,
                                                               const int32_t* __restrict__ arena,
                                                               uint32_t* __restrict__ cnt) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint64_t nwarps = (uint64_t)gridDim.x * (kCovThreads / 32);
    const uint64_t groups = (T + 31) / 32;
    for (uint64_t gidx = (uint64_t)blockIdx.x * (kCovThreads / 32) + wib; gidx < groups; gidx += nwarps) {
        const uint64_t j = gidx * 32 + lane;
        const bool valid = j < T;
        warp_members(valid ? h_off[j] : 0, valid ? h_len[j] : 0u, arena,
                     [&](int, int32_t u) { add_aggregated(cnt, u); });
    }
}

// cursor[u] starts at inv_off[u], so one atomic reserves an entry's final
// place (a counter from 0 also cost a scattered read of inv_off[u] an entry).
// Bound by the returning atomics, one an entry, and by their latency: four
// runs of members in flight. Whole build, with the scan of the counts, at
// 200K-5M samples: triangle Chung-Lu .68 -> .67 ms and weighted cascade
// 1.36 -> 1.30 from one run to four; .42 -> .33 on a 4M-vertex graph.
__global__ void __launch_bounds__(kCovThreads) k_fill_inverted(const uint64_t* __restrict__ h_off,
                                                               const uint32_t* __restrict__ h_len, uint64_t T,
                                                               const int32_t* __restrict__ arena,
                                                               unsigned long long* __restrict__ cursor,
                                                               uint32_t* __restrict__ inv) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint64_t nwarps = (uint64_t)gridDim.x * (kCovThreads / 32);
    const uint64_t groups = (T + 31) / 32;
    for (uint64_t gidx = (uint64_t)blockIdx.x * (kCovThreads / 32) + wib; gidx < groups; gidx += nwarps) {
        const uint64_t j0 = gidx * 32;
        const uint64_t j = j0 + lane;
        const bool valid = j < T;
        warp_members<kFillRuns>(valid ? h_off[j] : 0, valid ? h_len[j] : 0u, arena, [&](int owner, int32_t u) {
            inv[atomicAdd(&cursor[u], 1ull)] = (uint32_t)(j0 + owner);
        });
    }
}

struct KeyId {
    u128 key;
    uint32_t id;
    uint32_t valid;
};

__device__ __forceinline__ bool better(const KeyId& a, const KeyId& b) {
    if (a.valid != b.valid) return a.valid > b.valid;
    if (a.key != b.key) return a.key > b.key;
    return a.id < b.id;
}

__device__ __forceinline__ KeyId shfl_down_keyid(const KeyId& x, int d) {
    KeyId y;
    y.key = shfl_down_u128(x.key, d);
    y.id = __shfl_down_sync(kFull, x.id, d);
    y.valid = __shfl_down_sync(kFull, x.valid, d);
    return y;
}

__device__ KeyId block_best(KeyId b, KeyId* s_part) {
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const KeyId o = shfl_down_keyid(b, d);
        if (better(o, b)) b = o;
    }
    if (lane == 0) s_part[wib] = b;
    __syncthreads();
    if (wib == 0) {
        b = lane < (int)(blockDim.x / 32) ? s_part[lane] : KeyId{0, 0xFFFFFFFFu, 0};
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const KeyId o = shfl_down_keyid(b, d);
            if (better(o, b)) b = o;
        }
    }
    return b;  // valid in thread 0
}

// One candidate of the greedy argmax: the exact key Delta W + T (2^f - w)
// (below 2^94: T < 2^32, W <= 2^61) in three words, the vertex (~0: none),
// its Delta, and its inverted list where the holder knows it.
struct __align__(16) Cand {
    uint32_t k2, k1, k0, id;
    uint32_t d, cnt;
    uint64_t lo;
};
constexpr uint32_t kNone = 0xFFFFFFFFu;

__device__ __forceinline__ Cand no_cand() { return Cand{0, 0, 0, kNone, 0, 0, 0}; }

__device__ __forceinline__ bool cand_better(const Cand& a, const Cand& b) {  // larger key, then lower id
    if (a.k2 != b.k2) return a.k2 > b.k2;
    if (a.k1 != b.k1) return a.k1 > b.k1;
    if (a.k0 != b.k0) return a.k0 > b.k0;
    return a.id < b.id;
}

// The lane that holds the warp's best candidate, by word-wise reductions.
__device__ __forceinline__ int warp_best_lane(const Cand& c) {
    const uint32_t m2 = __reduce_max_sync(kFull, c.k2);
    bool e = c.k2 == m2;
    const uint32_t m1 = __reduce_max_sync(kFull, e ? c.k1 : 0u);
    e = e && c.k1 == m1;
    const uint32_t m0 = __reduce_max_sync(kFull, e ? c.k0 : 0u);
    e = e && c.k0 == m0;
    const uint32_t id = __reduce_min_sync(kFull, e ? c.id : kNone);
    return __ffs(__ballot_sync(kFull, e && c.id == id)) - 1;
}

__device__ __forceinline__ Cand ldcg_cand(const Cand* p) {
    const uint4* q = reinterpret_cast<const uint4*>(p);
    const uint4 x = __ldcg(q), y = __ldcg(q + 1);
    return Cand{x.x, x.y, x.z, x.w, y.x, y.y, (uint64_t)y.z | ((uint64_t)y.w << 32)};
}

// Control words of one greedy call, zero at its start.
struct GreedyCtl {
    unsigned int arrived;  // grid barrier arrivals
    unsigned int pool_n;
    unsigned int gave_up;  // a barrier wait ran out (it cannot while every block runs)
    unsigned int pad[29];
    unsigned int reached;  // the last grid barrier that every block arrived at, on a line of its own
    unsigned int pad2[31];
};

struct GreedyArgs {
    const uint64_t* w;
    uint8_t* inS;
    uint32_t* delta;
    int64_t n;
    uint64_t W, T;
    double ratio;     // T / W, for the pool's buckets
    int f;
    int32_t k;
    const uint64_t* inv_off;
    const uint32_t* inv;
    const uint64_t* h_off;
    const uint32_t* h_len;
    const int32_t* arena;
    uint32_t* covered;
    Cand* partial;
    Cand* seg_best;   // per segment of kGreedySeg vertices: its best of the last scan
    int64_t nseg;
    uint32_t* pool;   // kGreedyThreads vertices
    uint32_t* hist;   // kBuckets counters of the vertices by rounded key (k_greedy_init)
    GreedyCtl* ctl;
    int32_t* seeds;
    int64_t* cov_out;
    double* est_out;
    int ris;
};

// All k rounds of Alg. 3 in one cooperative launch, one block per SM. A round
// is a chain of memory latencies and grid barriers far more than it is work,
// so:
//   - The argmax comes from a pool: the vertices outside S with the largest
//     keys, up to one a thread, which every block holds alike, and the exact
//     best key outside the pool. Keys only decrease, so while the pool's best
//     beats that bound it is the argmax (ties to the lowest id), and every
//     block finds it by itself, with no exchange. When it no longer does, the
//     pool is refilled from all vertices (a histogram of rounded keys picks
//     how far down it goes; a vertex that does not get in bounds it, so that
//     membership decides nothing but speed).
//   - Where too many vertices tie for a pool, rounds scan segments of 256
//     vertices instead: a segment whose best is still outside S with an
//     unchanged Delta keeps it, the others are rescanned, one warp each.
//   - A block may change Delta only after every block has read it; that grid
//     barrier is entered before the walk and left after the walk's first
//     loads (list, covered bits, headers), which do not touch Delta.
//   - The walk: a thread takes an entry of the winner's inverted list, and the
//     members of the block's uncovered samples are dealt to its threads end
//     to end, whatever their sizes.
// Data that other blocks change during the launch is read through L2
// (ld.global.cg), never from a possibly stale L1 line.
// Chung-Lu 1M / 17.5M WC, 1M samples, k = 1000: 20 -> 8 ms, 8 us a round, of
// which the grid barrier at its end 3 us, the argmax 1.8 us, the list and the
// headers 1.7 us, the members 1.2 us (the argmax over the segments with two
// grid barriers a round, each list run of 32 entries on one warp, before).
constexpr int kGreedyThreads = 1024;
constexpr int kGreedySegLog = 8;  // vertices per segment: 256
constexpr int64_t kGreedySeg = 1ll << kGreedySegLog;
constexpr int kBuckets = 8192;           // exponent and five mantissa bits of a rounded key / W
constexpr uint32_t kPoolMin = 64;        // a smaller pool does not pay for its refill
constexpr uint32_t kSegRounds = 64;      // segment rounds before a pool is tried again
constexpr unsigned int kBarSpins = 1u << 23;  // polls of a grid barrier before giving up (~10 s)

// key / W, rounded: where a vertex stands in the pool's histogram
__device__ __forceinline__ uint32_t greedy_bucket(uint32_t d, uint64_t gap, double ratio, int ris) {
    const float x = ris ? (float)d : (float)((double)d + (double)gap * ratio);
    return __float_as_uint(x) >> 18;
}

// Delta_R(v, {}) = number of samples containing v = length of v's list, and
// the histogram of the first pool.
__global__ void __launch_bounds__(kGreedyThreads) k_greedy_init(GreedyArgs a) {
    __shared__ uint32_t s_hist[kBuckets];
    for (int i = threadIdx.x; i < kBuckets; i += kGreedyThreads) s_hist[i] = 0;
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * kGreedyThreads;
    for (int64_t v0 = (int64_t)blockIdx.x * kGreedyThreads + (threadIdx.x & ~31); v0 < a.n; v0 += stride) {
        const int64_t v = v0 + (threadIdx.x & 31);
        uint32_t b = kBuckets;
        if (v < a.n) {
            const uint32_t d = (uint32_t)(a.inv_off[v + 1] - a.inv_off[v]);
            a.delta[v] = d;
            b = greedy_bucket(d, (1ull << a.f) - a.w[v], a.ratio, a.ris);
        }
        // most vertices share a few low buckets: one atomic a warp for each
        const unsigned peers = __match_any_sync(kFull, b);
        if (b < kBuckets && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&s_hist[b], (uint32_t)__popc(peers));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kBuckets; i += kGreedyThreads)
        if (s_hist[i]) atomicAdd(&a.hist[i], s_hist[i]);
}

// Grid barrier in two halves (the grid is launched cooperatively): an arrival
// is one atomic a block, the last of them publishes the barrier's number, and
// one thread a block polls that word. Few pollers and no sequentially
// consistent fence: with every block polling a word of every other, or with
// __threadfence() at each end, a barrier took 9,000 to 17,000 cycles, with the
// cooperative-groups one 9,000, with this one 5,900 (800 where the walk's
// first loads hide it).
struct GridBar {
    GreedyCtl* ctl;
    uint32_t* failed;  // shared
    uint32_t goal;

    // After a block barrier. ordered: the block's writes before it are seen by
    // the other blocks after their wait (else only its reads are over).
    __device__ __forceinline__ void arrive(bool ordered) {
        ++goal;
        if (threadIdx.x != 0) return;
        uint32_t old;
        if (ordered) {
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(&ctl->arrived) : "memory");
            if (old + 1u == goal * gridDim.x)
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&ctl->reached), "r"(goal) : "memory");
        } else {
            asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(&ctl->arrived) : "memory");
            if (old + 1u == goal * gridDim.x)
                asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(&ctl->reached), "r"(goal) : "memory");
        }
    }
    // false: the wait ran out
    __device__ __forceinline__ bool wait(bool ordered) {
        if (threadIdx.x == 0) {
            uint32_t x;
            for (uint32_t spins = 0;;) {
                if (ordered)
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(&ctl->reached) : "memory");
                else
                    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(&ctl->reached) : "memory");
                if ((int)(x - goal) >= 0) break;
                if (++spins > kBarSpins) {
                    atomicOr(&ctl->gave_up, 1u);
                    *failed = 1;
                    break;
                }
            }
        }
        __syncthreads();
        return *failed == 0;
    }
    __device__ __forceinline__ bool sync() {
        __syncthreads();
        arrive(true);
        return wait(true);
    }
};

__global__ void __launch_bounds__(kGreedyThreads, 1) k_greedy_rounds(GreedyArgs a) {
    __shared__ Cand s_part[2][kGreedyThreads / 32];
    __shared__ __align__(16) uint32_t s_hist[kBuckets];  // a refill's histogram, or
    uint64_t* const s_off = reinterpret_cast<uint64_t*>(s_hist);  // the walk's samples: arena offset,
    uint64_t* const s_end = s_off + kGreedyThreads;               // and members of the block up to its end
    static_assert(kBuckets * sizeof(uint32_t) >= 2 * kGreedyThreads * sizeof(uint64_t), "the walk's arrays fit");
    __shared__ uint32_t s_hkey[kHotSlots], s_hcnt[kHotSlots];
    __shared__ uint64_t s_wsum[kGreedyThreads / 32];
    __shared__ uint32_t s_cut, s_failed;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint64_t one_f = 1ull << a.f;
    const int nw = kGreedyThreads / 32;
    for (int i = threadIdx.x; i < kHotSlots; i += blockDim.x) {
        s_hkey[i] = kHotEmpty;
        s_hcnt[i] = 0;
    }
    if (threadIdx.x == 0) s_failed = 0;
    GridBar bar{a.ctl, &s_failed, 0u};
    int par = 0;  // half of s_part of the next block reduction

    auto make = [&](uint32_t v, uint32_t d, uint64_t w) -> Cand {
        const u128 key = a.ris ? (u128)d : (u128)d * a.W + (u128)a.T * (one_f - w);
        return Cand{(uint32_t)(key >> 64), (uint32_t)(key >> 32), (uint32_t)key, v, d, 0u, 0ull};
    };
    // the block's best of the threads' candidates, known to every thread; a
    // block barrier stands between the candidates' loads and the return
    auto block_cand = [&](const Cand& c) -> Cand {
        const int src = warp_best_lane(c);
        if (lane == src) s_part[par][wib] = c;
        __syncthreads();
        const int win = warp_best_lane(s_part[par][lane]);
        const Cand r = s_part[par][win];
        par ^= 1;
        return r;
    };
    // the grid's best, known to every thread (one grid barrier). false, here and
    // from its callers: a barrier's wait ran out, so that other blocks' writes may
    // be missing; nothing is read by them, the block ends
    auto grid_cand = [&](const Cand& c, Cand* best) -> bool {
        const Cand b = block_cand(c);
        if (threadIdx.x == 0) a.partial[blockIdx.x] = b;
        if (!bar.sync()) return false;
        Cand r = no_cand();
        for (unsigned i = lane; i < gridDim.x; i += 32) {
            const Cand x = ldcg_cand(a.partial + i);
            if (cand_better(x, r)) r = x;
        }
        const int src = warp_best_lane(r);
        r.k2 = __shfl_sync(kFull, r.k2, src);
        r.k1 = __shfl_sync(kFull, r.k1, src);
        r.k0 = __shfl_sync(kFull, r.k0, src);
        r.id = __shfl_sync(kFull, r.id, src);
        r.d = __shfl_sync(kFull, r.d, src);
        *best = r;
        return true;
    };
    auto bucket = [&](uint32_t d, uint64_t w) { return greedy_bucket(d, one_f - w, a.ratio, a.ris); };

    // the pool entry of this thread
    uint32_t p_id = kNone, p_cnt = 0;
    uint64_t p_w = 0, p_lo = 0;
    auto pool_best = [&]() -> Cand {
        Cand c = no_cand();
        if (p_id != kNone) {
            c = make(p_id, __ldcg(a.delta + p_id), p_w);
            c.cnt = p_cnt;
            c.lo = p_lo;
        }
        return block_cand(c);
    };
    // Fills the pool from the vertices outside S; *rest: the best of the others.
    bool hist_ready = true;  // k_greedy_init's
    auto refill = [&](Cand* rest) -> bool {
        const int64_t stride = (int64_t)gridDim.x * kGreedyThreads;
        const int64_t first = (int64_t)blockIdx.x * kGreedyThreads + threadIdx.x;
        if (threadIdx.x == 0) s_cut = kBuckets;
        __syncthreads();
        if (!hist_ready) {
            for (int i = threadIdx.x; i < kBuckets; i += kGreedyThreads) s_hist[i] = 0;
            __syncthreads();
            for (int64_t v0 = first - lane; v0 < a.n; v0 += stride) {  // warp-uniform
                const int64_t v = v0 + lane;
                uint32_t b = kBuckets;
                if (v < a.n && !__ldcg(a.inS + v)) b = bucket(__ldcg(a.delta + v), a.w[v]);
                const unsigned peers = __match_any_sync(kFull, b);
                if (b < kBuckets && lane == __ffs(peers) - 1) atomicAdd(&s_hist[b], (uint32_t)__popc(peers));
            }
            __syncthreads();
            for (int i = threadIdx.x; i < kBuckets; i += kGreedyThreads)
                if (s_hist[i]) atomicAdd(&a.hist[i], s_hist[i]);
            if (!bar.sync()) return false;
        }
        hist_ready = false;
        // the lowest bucket down to which the pool has room: thread t counts
        // buckets 8 (1023 - t) + 7 .. 8 (1023 - t), in descending order over t
        constexpr int kPer = kBuckets / kGreedyThreads;
        const int top = kPer * (kGreedyThreads - 1 - threadIdx.x) + kPer - 1;
        uint32_t c[kPer], sum = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            c[i] = __ldcg(a.hist + top - i);
            sum += c[i];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) s_wsum[wib] = incl;
        __syncthreads();
        uint32_t before = incl - sum;
        for (int q = 0; q < wib; ++q) before += (uint32_t)s_wsum[q];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            before += c[i];
            if (before <= (uint32_t)kGreedyThreads) atomicMin(&s_cut, (uint32_t)(top - i));
        }
        __syncthreads();
        const uint32_t cut = s_cut;
        Cand out = no_cand();
        for (int64_t v0 = first; v0 < a.n; v0 += 4 * stride) {  // four vertices a pass, their loads together
            uint8_t in4[4];
            uint32_t d4[4];
            uint64_t w4[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t v = v0 + q * stride;
                in4[q] = 1;
                if (v < a.n) {
                    in4[q] = __ldcg(a.inS + v);
                    d4[q] = __ldcg(a.delta + v);
                    w4[q] = a.w[v];
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (in4[q]) continue;
                const uint32_t v = (uint32_t)(v0 + q * stride);
                bool pooled = false;
                if (bucket(d4[q], w4[q]) >= cut) {
                    const uint32_t slot = atomicAdd(&a.ctl->pool_n, 1u);
                    pooled = slot < (uint32_t)kGreedyThreads;
                    if (pooled) a.pool[slot] = v;
                }
                // the others bound the pool, one that found it full (it cannot
                // while a key rounds alike here and in the histogram) included
                if (!pooled) {
                    const Cand x = make(v, d4[q], w4[q]);
                    if (cand_better(x, out)) out = x;
                }
            }
        }
        if (!grid_cand(out, rest)) return false;
        const uint32_t np = min(__ldcg(&a.ctl->pool_n), (uint32_t)kGreedyThreads);
        p_id = kNone;
        if (threadIdx.x < np) {
            p_id = __ldcg(a.pool + threadIdx.x);
            p_w = a.w[p_id];
            p_lo = a.inv_off[p_id];
            p_cnt = (uint32_t)(a.inv_off[p_id + 1] - p_lo);
        }
        return true;
    };
    // The best vertex outside S by segments. Warp gw of W takes segments
    // gw + W i, 32 of them at a time (lane l: gw + W (32 i + l)); the block
    // index varies fastest over gw, so a few segments already spread over
    // every SM.
    bool seg_init = false;
    auto seg_scan = [&](Cand* best) -> bool {
        Cand wbest = no_cand();
        const int64_t W = (int64_t)gridDim.x * nw, gw = (int64_t)wib * gridDim.x + blockIdx.x;
        for (int64_t g0 = gw; g0 < a.nseg; g0 += 32 * W) {
            const int64_t sg = g0 + lane * W;
            Cand b = no_cand();
            bool ok = sg >= a.nseg;
            if (!ok && seg_init) {
                b = ldcg_cand(a.seg_best + sg);
                ok = b.id == kNone || (!__ldcg(a.inS + b.id) && __ldcg(a.delta + b.id) == b.d);
            }
            unsigned redo = __ballot_sync(kFull, !ok);
            while (redo) {
                const int src = __ffs(redo) - 1;
                redo &= redo - 1;
                const int64_t v_lo = (g0 + src * W) << kGreedySegLog, v_hi = min(a.n, v_lo + kGreedySeg);
                Cand r = no_cand();
                // four of the lane's vertices per pass, their loads issued together
                for (int64_t v0 = v_lo + lane; v0 < v_hi; v0 += 128) {
                    uint8_t in4[4];
                    uint32_t d4[4];
                    uint64_t w4[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int64_t v = v0 + 32 * q;
                        in4[q] = 1;
                        if (v < v_hi) {
                            in4[q] = __ldcg(a.inS + v);
                            d4[q] = __ldcg(a.delta + v);
                            w4[q] = a.w[v];
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (in4[q]) continue;
                        const Cand c = make((uint32_t)(v0 + 32 * q), d4[q], w4[q]);
                        if (cand_better(c, r)) r = c;
                    }
                }
                const int top = warp_best_lane(r);
                r.k2 = __shfl_sync(kFull, r.k2, top);
                r.k1 = __shfl_sync(kFull, r.k1, top);
                r.k0 = __shfl_sync(kFull, r.k0, top);
                r.id = __shfl_sync(kFull, r.id, top);
                r.d = __shfl_sync(kFull, r.d, top);
                if (lane == src) b = r;
                if (lane == 0) a.seg_best[g0 + src * W] = r;
            }
            if (cand_better(b, wbest)) wbest = b;
        }
        seg_init = true;
        return grid_cand(wbest, best);
    };

    uint64_t cov = 0, sum_c = 0;  // running totals, kept by one thread
    bool pool_on = false;
    uint32_t seg_left = 0;
    Cand bound = no_cand();  // the best outside the pool when it was filled
    __syncthreads();
    for (int32_t round = 0; round < a.k; ++round) {
        Cand win = no_cand();
        bool found = false, refilled = false;
        if (pool_on) {
            win = pool_best();
            found = cand_better(win, bound);
        }
        if (!found && seg_left) {
            --seg_left;
            if (!seg_scan(&win)) return;  // the host reports it
        } else if (!found) {
            if (!refill(&bound)) return;
            refilled = true;
            win = pool_best();
            if (!cand_better(win, bound)) win = bound;
            pool_on = __syncthreads_count(p_id != kNone) >= (int)kPoolMin;
            if (!pool_on) seg_left = kSegRounds;
        }
        const uint32_t v = win.id;
        // every read of Delta in this block is done: changes may start once
        // all blocks are here
        bar.arrive(false);
        if (p_id == v) p_id = kNone;
        uint64_t lo = win.lo, cnt = win.cnt;
        if (cnt == 0) {  // not a pool entry's (or an empty list)
            lo = a.inv_off[v];
            cnt = a.inv_off[v + 1] - lo;
        }
        // the uncovered samples of the committed vertex, an entry a thread: a
        // list of up to one entry a thread of the grid is dealt over the blocks
        // entry by entry, a longer one in runs of 1024
        const bool spread = cnt <= (uint64_t)gridDim.x * kGreedyThreads;
        const uint64_t step = (uint64_t)gridDim.x * kGreedyThreads;
        for (uint64_t base = 0; base < cnt || base == 0; base += step) {
            const uint64_t x = spread ? (uint64_t)threadIdx.x * gridDim.x + blockIdx.x
                                      : base + (uint64_t)blockIdx.x * kGreedyThreads + threadIdx.x;
            uint64_t off = 0;
            uint32_t len = 0;
            if (x < cnt) {
                const uint32_t j = a.inv[lo + x];
                const uint32_t bit = 1u << (j & 31);
                const uint64_t o = a.h_off[j];  // with the bit, not after it
                const uint32_t l = a.h_len[j];
                if ((atomicOr(&a.covered[j >> 5], bit) & bit) == 0) {
                    off = o;
                    len = l;
                }
            }
            // the block's members end to end: inclusive prefix of the lengths
            uint64_t incl = len;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint64_t y = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += y;
            }
            if (lane == 31) s_wsum[wib] = incl;
            if (base == 0) {
                if (!bar.wait(false)) return;  // the host reports it
                if (refilled && blockIdx.x == 0) {  // every block has read these
                    for (int i = threadIdx.x; i < kBuckets; i += kGreedyThreads) a.hist[i] = 0;
                    if (threadIdx.x == 0) a.ctl->pool_n = 0;
                }
                // read (through L2) after the round's last grid barrier
                if (blockIdx.x == 0 && threadIdx.x == 0) a.inS[v] = 1;
            } else {
                __syncthreads();
            }
            uint64_t before = 0, total = 0;
            {
                uint64_t wsum = s_wsum[lane];
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint64_t y = __shfl_up_sync(kFull, wsum, d);
                    if (lane >= d) wsum += y;
                }
                total = __shfl_sync(kFull, wsum, 31);
                before = __shfl_sync(kFull, wsum, wib > 0 ? wib - 1 : 0);
                if (wib == 0) before = 0;
            }
            if (total) {
                s_off[threadIdx.x] = off - (before + incl - len);  // + a member's place in the block
                s_end[threadIdx.x] = before + incl;
                __syncthreads();
                for (uint64_t p = threadIdx.x; p < total; p += kGreedyThreads) {
                    int owner = 0;  // the sample that holds member p: entries that end at or before it
#pragma unroll
                    for (int b = kGreedyThreads / 2; b; b >>= 1)
                        if (s_end[owner + b - 1] <= p) owner += b;
                    sub_merged(a.delta, a.arena[s_off[owner] + p], s_hkey, s_hcnt);
                }
            }
            __syncthreads();  // s_wsum, s_off and s_end are free again
        }
        for (int i = threadIdx.x; i < kHotSlots; i += blockDim.x) {
            const uint32_t key = s_hkey[i];
            if (key != kHotEmpty) {
                atomicSub(&a.delta[key], s_hcnt[i]);
                s_hkey[i] = kHotEmpty;
                s_hcnt[i] = 0;
            }
        }
        __syncthreads();
        bar.arrive(true);
        if (blockIdx.x == 0 && threadIdx.x == kGreedyThreads - 1) {  // while the barrier is waited for
            cov += win.d;  // Delta_v as read, before any walk of this round
            sum_c += one_f - a.w[v];
            a.seeds[round] = (int32_t)v;
            a.cov_out[round] = (int64_t)cov;
            const u128 N = a.ris ? (u128)cov * (uint64_t)a.n : (u128)cov * a.W + (u128)a.T * sum_c;
            const u128 D = a.ris ? (u128)a.T : (u128)a.T << a.f;
            a.est_out[round] = u128_to_double(N) / u128_to_double(D);
        }
        if (!bar.wait(true)) return;  // the host reports it
    }
}

static int build_inverted(skis_sketch* s, cudaStream_t st, std::string* err) {
    const char* where = "inverted index";
    if (s->inv && s->inv_T == s->T) return SKIS_OK;
    const int64_t n = s->g->n;
    const uint64_t T = s->T;
    if (T >= (1ull << 32)) {
        *err = "inverted index: the sketch must hold fewer than 2^32 samples";
        return SKIS_EINVAL;
    }
    dev_free(s->inv, st);
    s->inv = nullptr;
    s->inv_T = 0;
    if (!s->inv_off) CV_CUDA(dev_alloc_t(&s->inv_off, (size_t)n + 1, st));
    uint64_t E = 0;
    const int cblocks = coverage_blocks(T);
    if (s->vcount && s->vcount_ok && s->vcount_T == T) {  // counted while sampling
        CV_CUDA(scan_u32_to_u64(s->vcount, s->inv_off, n, st));
    } else {
        uint32_t* cnt = nullptr;
        CV_CUDA(dev_alloc_t(&cnt, (size_t)n, st));
        cudaError_t e = cudaMemsetAsync(cnt, 0, (size_t)n * sizeof(uint32_t), st);
        if (e == cudaSuccess) {
            k_count_members<<<cblocks, kCovThreads, 0, st>>>(s->h_off, s->h_len, T, s->arena, cnt); note_launch();
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = scan_u32_to_u64(cnt, s->inv_off, n, st);
        dev_free(cnt, st);
        CV_CUDA(e);
    }
    CV_CUDA(cudaMemcpyAsync(&E, s->inv_off + n, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    CV_CUDA(cudaStreamSynchronize(st));
    CV_CUDA(dev_alloc_t(&s->inv, (size_t)std::max<uint64_t>(E, 1), st));
    unsigned long long* cursor = nullptr;
    CV_CUDA(dev_alloc_t(&cursor, (size_t)n, st));
    CV_CUDA(cudaMemcpyAsync(cursor, s->inv_off, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
    k_fill_inverted<<<cblocks, kCovThreads, 0, st>>>(s->h_off, s->h_len, T, s->arena, cursor, s->inv); note_launch();
    CV_CUDA(cudaGetLastError());
    dev_free(cursor, st);
    s->inv_T = T;
    return SKIS_OK;
}

int sketch_inverted(skis_sketch* s, cudaStream_t st, std::string* err) {
    return with_room(s, st, err, [&] { return build_inverted(s, st, err); });
}

constexpr int32_t kGreedyPacked = 4096;  // largest k whose results come back in one copy

int sketch_greedy(skis_sketch* s, int32_t k, int32_t* h_seeds, int64_t* h_cov, double* h_est, cudaStream_t st,
                  std::string* err) {
    const char* where = "skis_greedy_maxcover";
    const skis_graph* g = s->g;
    const int64_t n = g->n;
    const uint64_t T = s->T;
    if (k < 0 || k > n) {
        *err = "skis_greedy_maxcover: k must be in [0, n]";
        return SKIS_EINVAL;
    }
    if (T == 0 || T >= (1ull << 32)) {
        *err = "skis_greedy_maxcover: the sketch must hold between 1 and 2^32 - 1 samples";
        return SKIS_EINVAL;
    }
    if (k == 0) return SKIS_OK;
    int rc = sketch_inverted(s, st, err);
    if (rc != SKIS_OK) return rc;
    char* buf = nullptr;
    auto body = [&]() -> int {
        int per_sm = 0;
        CV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_greedy_rounds, kGreedyThreads, 0));
        if (per_sm < 1) {
            *err = "skis_greedy_maxcover: the cooperative kernel does not fit on an SM";
            return SKIS_ERR_CUDA;
        }
        const int gblocks = sm_count();  // one block per SM
        const int64_t nseg = (n + kGreedySeg - 1) / kGreedySeg;
        // one allocation, its first part zeroed at once, the control words and
        // the results next to one another for one copy back (each allocation or
        // copy more is some microseconds of a call that takes 150 on a small sketch)
        size_t bytes = 0;
        auto take = [&](size_t b) {
            const size_t at = bytes;
            bytes += (b + 127) & ~(size_t)127;
            return at;
        };
        const size_t at_hist = take(kBuckets * sizeof(uint32_t)), at_inS = take((size_t)n);
        const size_t at_covered = take((size_t)((T + 31) / 32) * sizeof(uint32_t));
        const size_t at_ctl = take(sizeof(GreedyCtl)), zeroed = bytes;
        const size_t at_est = take((size_t)k * sizeof(double)), at_cov = take((size_t)k * sizeof(int64_t));
        const size_t at_seeds = take((size_t)k * sizeof(int32_t)), copied = bytes - at_ctl;
        const size_t at_partial = take((size_t)gblocks * sizeof(Cand)), at_seg = take((size_t)nseg * sizeof(Cand));
        const size_t at_pool = take(kGreedyThreads * sizeof(uint32_t)), at_delta = take((size_t)n * sizeof(uint32_t));
        const bool packed = k <= kGreedyPacked;  // else straight to the caller's arrays
        const size_t out_bytes = packed ? copied : sizeof(GreedyCtl);
        // on the heap: the caller's thread may have little stack
        const std::unique_ptr<char[]> h_out(new (std::nothrow) char[out_bytes]);
        if (!h_out) {
            *err = "skis_greedy_maxcover: host allocation failed";
            return SKIS_ENOMEM;
        }
        const int room = with_room(s, st, err, [&]() -> int {
            CV_CUDA(dev_alloc_t(&buf, bytes, st));
            return SKIS_OK;
        });
        if (room != SKIS_OK) return room;
        CV_CUDA(cudaMemsetAsync(buf, 0, zeroed, st));
        GreedyArgs ga;
        ga.w = g->w;
        ga.inS = reinterpret_cast<uint8_t*>(buf + at_inS);
        ga.delta = reinterpret_cast<uint32_t*>(buf + at_delta);
        ga.n = n;
        ga.W = g->W;
        ga.T = T;
        ga.ratio = g->W ? (double)T / (double)g->W : 0.0;
        ga.f = g->f;
        ga.k = k;
        ga.inv_off = s->inv_off;
        ga.inv = s->inv;
        ga.h_off = s->h_off;
        ga.h_len = s->h_len;
        ga.arena = s->arena;
        ga.covered = reinterpret_cast<uint32_t*>(buf + at_covered);
        ga.partial = reinterpret_cast<Cand*>(buf + at_partial);
        ga.seg_best = reinterpret_cast<Cand*>(buf + at_seg);
        ga.nseg = nseg;
        ga.pool = reinterpret_cast<uint32_t*>(buf + at_pool);
        ga.hist = reinterpret_cast<uint32_t*>(buf + at_hist);
        ga.ctl = reinterpret_cast<GreedyCtl*>(buf + at_ctl);
        ga.seeds = reinterpret_cast<int32_t*>(buf + at_seeds);
        ga.cov_out = reinterpret_cast<int64_t*>(buf + at_cov);
        ga.est_out = reinterpret_cast<double*>(buf + at_est);
        ga.ris = s->ris;
        const int b1 = (int)std::max<int64_t>(1, std::min<int64_t>((n + kGreedyThreads - 1) / kGreedyThreads,
                                                                   (int64_t)sm_count() * 2));
        k_greedy_init<<<b1, kGreedyThreads, 0, st>>>(ga); note_launch();
        CV_CUDA(cudaGetLastError());
        void* kargs[] = {&ga};
        CV_CUDA(cudaLaunchCooperativeKernel((const void*)k_greedy_rounds, gblocks, kGreedyThreads, kargs, 0, st));
        note_launch();
        CV_CUDA(cudaMemcpyAsync(h_out.get(), buf + at_ctl, out_bytes, cudaMemcpyDeviceToHost, st));
        if (!packed) {
            CV_CUDA(cudaMemcpyAsync(h_seeds, ga.seeds, (size_t)k * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
            if (h_cov) CV_CUDA(cudaMemcpyAsync(h_cov, ga.cov_out, (size_t)k * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
            if (h_est) CV_CUDA(cudaMemcpyAsync(h_est, ga.est_out, (size_t)k * sizeof(double), cudaMemcpyDeviceToHost, st));
        }
        CV_CUDA(cudaStreamSynchronize(st));
        unsigned int gave_up = 0;
        std::memcpy(&gave_up, h_out.get() + offsetof(GreedyCtl, gave_up), sizeof(gave_up));
        if (gave_up) {
            *err = "skis_greedy_maxcover: internal error: a grid barrier ran out";
            return SKIS_ERR_INTERNAL;
        }
        if (packed) {
            std::memcpy(h_seeds, h_out.get() + (at_seeds - at_ctl), (size_t)k * sizeof(int32_t));
            if (h_cov) std::memcpy(h_cov, h_out.get() + (at_cov - at_ctl), (size_t)k * sizeof(int64_t));
            if (h_est) std::memcpy(h_est, h_out.get() + (at_est - at_ctl), (size_t)k * sizeof(double));
        }
        return SKIS_OK;
    };
    rc = body();
    dev_free(buf, st);
    return rc;
}

}  // namespace skis

// ------------------------------------------------------ sharded sketch
// A sketch split by sample id over ranks (every rank holds the samples of
// one id range of one seed's sketch). Coverage counts and Delta are sums
// over the ranks' samples, so the per-rank values are summed through the
// caller's all-reduce in a caller-owned device buffer, and every rank then
// takes the same decisions as one process holding the union sketch.
namespace skis {

__global__ void k_shard_delta0(const uint64_t* __restrict__ inv_off, int64_t n, int64_t* __restrict__ x) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += (int64_t)gridDim.x * blockDim.x)
        x[v] = v < n ? (int64_t)(inv_off[v + 1] - inv_off[v]) : 0;
}

// Block bests of the exact key Delta W + T (2^f - w_v) (RIS: Delta) over v
// outside S, ties to the lowest id.
__global__ void __launch_bounds__(256) k_shard_argmax(const int64_t* __restrict__ delta, const uint64_t* __restrict__ w,
                                                      const uint8_t* __restrict__ inS, int64_t n, uint64_t W,
                                                      uint64_t T, int f, int ris, KeyId* __restrict__ partial) {
    __shared__ KeyId s_part[256 / 32];
    const uint64_t one_f = 1ull << f;
    KeyId best{0, 0xFFFFFFFFu, 0};
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        if (inS[v]) continue;
        const u128 dv = (u128)(uint64_t)delta[v];
        const KeyId c{ris ? dv : dv * W + (u128)T * (one_f - w[v]), (uint32_t)v, 1u};
        if (better(c, best)) best = c;
    }
    best = block_best(best, s_part);
    if (threadIdx.x == 0) partial[blockIdx.x] = best;
}

// The round's winner from the block bests: joins S; recorded as seed r.
__global__ void k_shard_commit(const KeyId* __restrict__ partial, int nparts, uint8_t* __restrict__ inS,
                               int32_t* __restrict__ seeds, int32_t r, uint32_t* __restrict__ win) {
    const int lane = threadIdx.x & 31;
    KeyId b{0, 0xFFFFFFFFu, 0};
    for (int i = lane; i < nparts; i += 32)
        if (better(partial[i], b)) b = partial[i];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const KeyId o = shfl_down_keyid(b, d);
        if (better(o, b)) b = o;
    }
    if (lane == 0) {  // a valid winner exists: k <= n and each round adds one vertex
        inS[b.id] = 1;
        seeds[r] = (int32_t)b.id;
        *win = b.id;
    }
}

// Cover this rank's uncovered samples of the winner: x[u] += 1 for every
// member u of each, x[n] += the number of them.
__global__ void __launch_bounds__(256) k_shard_cover(const uint32_t* __restrict__ win,
                                                     const uint64_t* __restrict__ inv_off,
                                                     const uint32_t* __restrict__ inv,
                                                     const uint64_t* __restrict__ h_off,
                                                     const uint32_t* __restrict__ h_len,
                                                     const int32_t* __restrict__ arena, uint32_t* __restrict__ covered,
                                                     int64_t n, int64_t* __restrict__ x) {
    const int lane = threadIdx.x & 31;
    const uint32_t v = *win;
    const uint64_t lo = inv_off[v], cnt = inv_off[v + 1] - lo;
    const uint64_t nwarps = (uint64_t)gridDim.x * (blockDim.x / 32);
    unsigned long long* xc = reinterpret_cast<unsigned long long*>(x);
    for (uint64_t base = ((uint64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5)) * 32; base < cnt;
         base += nwarps * 32) {
        uint64_t off = 0;
        uint32_t len = 0;
        if (base + lane < cnt) {
            const uint32_t j = inv[lo + base + lane];
            const uint32_t bit = 1u << (j & 31);
            if ((atomicOr(&covered[j >> 5], bit) & bit) == 0) {
                off = h_off[j];
                len = h_len[j];
                atomicAdd(xc + n, 1ull);
            }
        }
        warp_members(off, len, arena, [&](int, int32_t u) { atomicAdd(xc + u, 1ull); });
    }
}

// Delta -= the summed decrements; the running coverage and Eq. 21 of the
// prefix S (thread 0; acc = {Cov, sum over S of 2^f - w_v}).
__global__ void k_shard_update(int64_t* __restrict__ delta, const int64_t* __restrict__ x, int64_t n,
                               const uint32_t* __restrict__ win, const uint64_t* __restrict__ w, uint64_t W,
                               uint64_t T, int f, int ris, int32_t r, uint64_t* __restrict__ acc,
                               int64_t* __restrict__ cov_out, double* __restrict__ est_out) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        delta[v] -= x[v];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const uint64_t cov = acc[0] + (uint64_t)x[n];
        const uint64_t sum_c = acc[1] + ((1ull << f) - w[*win]);
        acc[0] = cov;
        acc[1] = sum_c;
        cov_out[r] = (int64_t)cov;
        const u128 N = ris ? (u128)cov * (uint64_t)n : (u128)cov * W + (u128)T * sum_c;
        const u128 D = ris ? (u128)T : (u128)T << f;
        est_out[r] = u128_to_double(N) / u128_to_double(D);
    }
}

// The caller's all-reduce of buf[0, count), after the work that wrote it.
static int exchange(skis_allreduce_fn fn, void* ctx, int64_t* buf, int64_t count, cudaStream_t st, const char* where,
                    std::string* err) {
    const cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        *err = std::string(where) + ": CUDA error: " + cudaGetErrorString(e);
        return SKIS_ERR_CUDA;
    }
    if (fn(ctx, buf, count, (void*)st) != 0) {
        *err = std::string(where) + ": the all-reduce callback failed";
        return SKIS_ERR_EXCHANGE;
    }
    return SKIS_OK;
}

int sketch_estimate_sharded(skis_sketch* s, int32_t q, const int64_t* d_off, const int32_t* d_seeds,
                            const int64_t* h_off, int64_t* d_cov, double* d_est, int64_t* exch, skis_allreduce_fn fn,
                            void* ctx, cudaStream_t st, std::string* err) {
    const char* where = "skis_estimate_sharded";
    const skis_graph* g = s->g;
    double* tmp = nullptr;
    CV_CUDA(dev_alloc_t(&tmp, (size_t)q, st));
    // this rank's counts into exch[0, q) (validating the queries), its T into exch[q]
    int rc = sketch_estimate(s, q, d_off, d_seeds, h_off, exch, tmp, st, err);
    dev_free(tmp, st);
    if (rc != SKIS_OK) return rc;
    const int64_t T_rank = (int64_t)s->T;
    CV_CUDA(cudaMemcpyAsync(exch + q, &T_rank, sizeof(int64_t), cudaMemcpyHostToDevice, st));
    rc = exchange(fn, ctx, exch, (int64_t)q + 1, st, where, err);
    if (rc != SKIS_OK) return rc;
    int64_t T = 0;
    CV_CUDA(cudaMemcpyAsync(&T, exch + q, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CV_CUDA(cudaStreamSynchronize(st));
    for (int32_t q0 = 0; q0 < q; q0 += 64) {
        const int32_t qn = std::min<int32_t>(64, q - q0);
        k_estimate<<<div_up((int64_t)qn * 32, 256), 256, 0, st>>>(
            d_off, d_seeds, q0, qn, g->n, g->w, g->f, g->W, (uint64_t)T,
            reinterpret_cast<const unsigned long long*>(exch + q0), d_cov, d_est, s->ris);
        note_launch();
        CV_CUDA(cudaGetLastError());
    }
    CV_CUDA(cudaStreamSynchronize(st));
    return SKIS_OK;
}

int sketch_greedy_sharded(skis_sketch* s, int32_t k, int32_t* h_seeds, int64_t* h_cov, double* h_est, int64_t* exch,
                          skis_allreduce_fn fn, void* ctx, cudaStream_t st, std::string* err) {
    const char* where = "skis_greedy_maxcover_sharded";
    const skis_graph* g = s->g;
    const int64_t n = g->n;
    if (k < 0 || k > n) {
        *err = "skis_greedy_maxcover_sharded: k must be in [0, n]";
        return SKIS_EINVAL;
    }
    if (s->T >= (1ull << 32)) {
        *err = "skis_greedy_maxcover_sharded: a rank's sketch must hold fewer than 2^32 samples";
        return SKIS_EINVAL;
    }
    if (k == 0) return SKIS_OK;
    // the union sketch's T
    const int64_t T_rank = (int64_t)s->T;
    CV_CUDA(cudaMemcpyAsync(exch, &T_rank, sizeof(int64_t), cudaMemcpyHostToDevice, st));
    int rc = exchange(fn, ctx, exch, 1, st, where, err);
    if (rc != SKIS_OK) return rc;
    int64_t T = 0;
    CV_CUDA(cudaMemcpyAsync(&T, exch, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CV_CUDA(cudaStreamSynchronize(st));
    if (T <= 0) {
        *err = "skis_greedy_maxcover_sharded: the ranks' sketches hold no samples";
        return SKIS_EINVAL;
    }
    rc = sketch_inverted(s, st, err);
    if (rc != SKIS_OK) return rc;
    int64_t* delta = nullptr;
    uint8_t* inS = nullptr;
    uint32_t *covered = nullptr, *win = nullptr;
    KeyId* partial = nullptr;
    int32_t* d_seeds = nullptr;
    int64_t* d_cov = nullptr;
    double* d_est = nullptr;
    uint64_t* acc = nullptr;
    const int nb = sm_count() * 4;
    const uint64_t cwords = std::max<uint64_t>(1, (s->T + 31) / 32);
    auto body = [&]() -> int {
        int e = with_room(s, st, err, [&]() -> int {
            if (!delta) CV_CUDA(dev_alloc_t(&delta, (size_t)n, st));
            if (!inS) CV_CUDA(dev_alloc_t(&inS, (size_t)n, st));
            if (!covered) CV_CUDA(dev_alloc_t(&covered, (size_t)cwords, st));
            if (!win) CV_CUDA(dev_alloc_t(&win, 1, st));
            if (!partial) CV_CUDA(dev_alloc_t(&partial, (size_t)nb, st));
            if (!d_seeds) CV_CUDA(dev_alloc_t(&d_seeds, (size_t)k, st));
            if (!d_cov) CV_CUDA(dev_alloc_t(&d_cov, (size_t)k, st));
            if (!d_est) CV_CUDA(dev_alloc_t(&d_est, (size_t)k, st));
            if (!acc) CV_CUDA(dev_alloc_t(&acc, 2, st));
            return SKIS_OK;
        });
        if (e != SKIS_OK) return e;
        CV_CUDA(cudaMemsetAsync(inS, 0, (size_t)n, st));
        CV_CUDA(cudaMemsetAsync(covered, 0, cwords * sizeof(uint32_t), st));
        CV_CUDA(cudaMemsetAsync(acc, 0, 2 * sizeof(uint64_t), st));
        // Delta_R(v, {}) over the union: the ranks' list lengths summed
        const int b1 = (int)std::max<int64_t>(1, std::min<int64_t>((n + 256) / 256, (int64_t)sm_count() * 8));
        k_shard_delta0<<<b1, 256, 0, st>>>(s->inv_off, n, exch); note_launch();
        CV_CUDA(cudaGetLastError());
        e = exchange(fn, ctx, exch, n + 1, st, where, err);
        if (e != SKIS_OK) return e;
        CV_CUDA(cudaMemcpyAsync(delta, exch, (size_t)n * sizeof(int64_t), cudaMemcpyDeviceToDevice, st));
        const int cb = (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)sm_count() * 8, (s->T + 255) / 256));
        for (int32_t r = 0; r < k; ++r) {
            k_shard_argmax<<<nb, 256, 0, st>>>(delta, g->w, inS, n, g->W, (uint64_t)T, g->f, s->ris, partial);
            note_launch();
            k_shard_commit<<<1, 32, 0, st>>>(partial, nb, inS, d_seeds, r, win); note_launch();
            CV_CUDA(cudaMemsetAsync(exch, 0, (size_t)(n + 1) * sizeof(int64_t), st));
            k_shard_cover<<<cb, 256, 0, st>>>(win, s->inv_off, s->inv, s->h_off, s->h_len, s->arena, covered, n, exch);
            note_launch();
            CV_CUDA(cudaGetLastError());
            e = exchange(fn, ctx, exch, n + 1, st, where, err);
            if (e != SKIS_OK) return e;
            k_shard_update<<<b1, 256, 0, st>>>(delta, exch, n, win, g->w, g->W, (uint64_t)T, g->f, s->ris, r, acc,
                                               d_cov, d_est);
            note_launch();
            CV_CUDA(cudaGetLastError());
        }
        CV_CUDA(cudaMemcpyAsync(h_seeds, d_seeds, (size_t)k * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        if (h_cov) CV_CUDA(cudaMemcpyAsync(h_cov, d_cov, (size_t)k * sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        if (h_est) CV_CUDA(cudaMemcpyAsync(h_est, d_est, (size_t)k * sizeof(double), cudaMemcpyDeviceToHost, st));
        CV_CUDA(cudaStreamSynchronize(st));
        return SKIS_OK;
    };
    rc = body();
    dev_free(delta, st);
    dev_free(inS, st);
    dev_free(covered, st);
    dev_free(win, st);
    dev_free(partial, st);
    dev_free(d_seeds, st);
    dev_free(d_cov, st);
    dev_free(d_est, st);
    dev_free(acc, st);
    return rc;
}

}  // namespace skis
