// Importance Influence Sampling (Sec. III, Alg. 1) on the device, in three
// tiers chained by sample id.
//
// Lane tier (first): one lane per sample; each step draws one edge quad of
// the lane's current row (one Philox block = the 4 coins of a quad). Member
// lists (which are also Alg. 1's FIFO queues Q = members[head .. len)) hold
// up to 32 vertices per sample in shared memory; the row of the next pop is
// loaded ahead; finished samples are written out and lanes refilled in
// batches. A sample whose list outgrows it, that meets an in-row longer than
// the degree threshold, or that uses up its step or retry budget is handed
// by id to the warp tier.
//
// Warp tier: one warp per sample. The member list (256 entries) and an
// open-addressing hash set (the visited set R_j) live in shared memory; a
// larger sample moves to the warp's slot in global memory (1536 or 4096
// members). Edges of up to 32 queued vertices are spread over the lanes one
// edge quad at a time. A sample that outgrows it is handed, by id, to the CTA
// tier.
//
// CTA tier: one block per sample with a global n-bit visited bitmap and an
// n-entry global queue per block slot.
//
// All tiers compute the same R_j: every coin is a pure function of
// (seed, sample id, domain, round, edge), so R_j is the reverse-reachable set
// of the source in one live-edge world, whatever the order of expansion.
#include <algorithm>
#include <string>

#include "../../include/skis.h"
#include "skis_internal.cuh"

namespace skis {

constexpr int kWarpThreads = 256;  // 8 warps per block
constexpr int kQCap = 256;         // warp-tier members held in shared memory
constexpr int kHashBits = 9;
constexpr int kHCap = 1 << kHashBits;  // their hash slots (load <= 1/2 + one insert round)
constexpr int kIdBatch = 16;       // most sample ids a warp takes per work-cursor atomic
// Members a sample may have in the warp tier, past kQCap in the warp's global
// spill slot, and the slot's hash bits (load at most 1/2). The longest samples
// that are still narrow (a few rows a level) belong here, where 32 of them
// share an SM, and not on the CTA tier, where at most eight do: on Chung-Lu 1M /
// 17.5M WC (levels of 13 rows; four blocks an SM then) the two tiers take
// 10.6 ms with 1536 members and 7.5 ms with 4096. Speed does not set the line
// for small graphs: 100K samples of ER graphs of average in-degree 10 WC take,
// with 1536 / 4096 members, .79 / .78 ms at 5k vertices, 1.19 / .95 at 10k, 1.37
// / 1.03 at 20k and 1.96 / 1.96 at 50k (400K samples: 2.18 / 2.17, 2.77 / 2.48, 3.64 /
// 2.95, 5.50 / 4.34). The smaller slot keeps the CTA tier in use at the default
// split on graphs whose samples are compared whole, member by member, with the
// oracle's (test_er_workload_full_parity asks for samples of all three tiers).
struct SpillSize {
    uint32_t cap, hash_bits;
};
inline SpillSize spill_size(int64_t n) { return n >= 6 * 4096 ? SpillSize{4096, 13} : SpillSize{1536, 12}; }
constexpr int kRing = 64;          // queued members whose in-rows wait in shared memory
constexpr int kPend = 32 + 128;    // live edges waiting for an insert round: under 32, plus one quad a lane
// entries reserved per arena atomic; once a warp's reservation did not fit it
// asks for no more than it needs, so that the arena cursor ends at the demand
constexpr uint32_t kArenaChunk = 2048;        // warp tier
constexpr uint32_t kLaneArenaChunk = 512;     // lane tiers
constexpr uint32_t kEmpty = 0xFFFFFFFFu;

struct SampleArgs {
    const AliasEntry* __restrict__ alias;
    const RowInfo* __restrict__ rows;
    const int32_t* __restrict__ src;
    const uint32_t* __restrict__ tau;  // nullptr: thresholds are per row
    uint64_t n, W, seed;
    PhiloxKeys rk;                     // the round keys of seed
    uint32_t retry_cap;
    uint32_t max_deg;                  // thread tier: longest in-row it expands
    uint32_t max_steps;                // thread tier: edge quads per sample before handing it on
    uint32_t max_retries;              // thread tier: rejected rounds before handing it on
    uint32_t warp_max_coins;           // warp tier: in-edges a BFS may draw before handing it on
    uint32_t cta_hub_quads;            // CTA tier: edge quads that make a row a hub (0 = no hub loop)
    int ris;                           // plain RIS: uniform source, one unconditioned round
    // input ids: first_id + t (ids == nullptr) or ids[t], t < count (or
    // t < *count_dev when the list was filled by the previous tier)
    const uint64_t* ids;
    uint64_t first_id, count;
    const unsigned long long* count_dev;
    uint64_t id_base;                  // sample id of the sketch's first header (headers are indexed j - id_base)
    unsigned long long* work;          // id cursor of this launch
    uint64_t* out_ids;                 // samples handed to the next tier
    unsigned long long* out_count;
    uint64_t* ovf_ids;                 // samples whose arena reservation did not fit
    unsigned long long* novf;
    unsigned long long* arena_cursor;
    uint64_t* h_off;
    uint32_t* h_len;
    uint32_t* h_src;
    uint32_t* h_retries;
    uint64_t* h_coins;
    int32_t* arena;
    uint64_t arena_cap;
    DevStatus* status;
    uint32_t* bitmaps;
    uint32_t* slot_clean;    // CTA tier: the slot's bitmap has been cleared
    int32_t* queues;
    uint64_t bitmap_words;
    uint32_t queue_cap;      // CTA tier: entries of a slot's queue (also the slots' stride); a sample
                             // with more members is handed to a pass with n-entry queues
    const uint4* srcrec;  // lane tier: source record per input t (k_sources)
    const uint2* srcpick; // lane tier, bucket form: (picked in-edge, its source) per input t
    const uint64_t* lt_cum;  // LT graphs with per-edge thresholds: running weight sums, else nullptr
    const uint64_t* chain;   // bucket first step: the gamma chain per in-edge, else nullptr
    uint32_t* vcount;        // per-vertex member counts kept for the inverted index, or nullptr
    // the lane tier's prepass records for sample ids [up_first, up_first + up_count), which the
    // later tiers reuse for the samples handed on to them (nullptr: draw again)
    const uint4* up_rec;
    const uint2* up_pick;
    uint64_t up_first, up_count;
    // warp tier: a spill slot a warp, 2^hash_bits table words and cap members
    uint32_t* spill_hash;
    int32_t* spill_queue;
    SpillSize spill;
};


// a member written to the arena counts towards its vertex's list length
__device__ __forceinline__ void count_member(const SampleArgs& a, int32_t u) {
    if (a.vcount) atomicAdd(&a.vcount[u], 1u);
}

__device__ __forceinline__ uint64_t input_count(const SampleArgs& a) {
    return a.count_dev ? (uint64_t)*a.count_dev : a.count;
}

__device__ __forceinline__ uint64_t input_id(const SampleArgs& a, uint64_t t) {
    return a.ids ? a.ids[t] : a.first_id + t;
}

__device__ __forceinline__ void hand_on(const SampleArgs& a, uint64_t j) {
    const unsigned long long k = atomicAdd(a.out_count, 1ull);
    a.out_ids[k] = j;
}

__device__ __forceinline__ void arena_overflow(const SampleArgs& a, uint64_t j) {
    const unsigned long long k = atomicAdd(a.novf, 1ull);
    a.ovf_ids[k] = j;
    atomicOr(&a.status->flags, kStArena);
}

// Eq. probu through the alias table: column floor(U1 n), threshold draw
// floor(U2 W) from the SRC-domain block of sample j.
// (kSeedKey: the Philox keys advanced from the seed in registers, for a
// kernel whose occupancy the preloaded round keys would cut)
template <bool kSeedKey = false>
__device__ __forceinline__ uint32_t draw_source(const SampleArgs& a, uint64_t j) {
    const uint4 x = kSeedKey ? coin_block(a.seed, 0, 0, kDomSrc, j) : coin_block(a.rk, 0, 0, kDomSrc, j);
    const uint64_t u1 = (uint64_t)x.x | ((uint64_t)x.y << 32);
    const uint64_t u2 = (uint64_t)x.z | ((uint64_t)x.w << 32);
    const uint64_t col = __umul64hi(u1, a.n);
    if (a.ris) return (uint32_t)col;  // RIS: the uniform column alone
    const uint64_t y = __umul64hi(u2, a.W);
    const AliasEntry e = a.alias[col];
    return y < e.prob ? (uint32_t)col : e.alias;
}

// The bucket form of Alg. 1's conditioned first step (Eq. probn): bucket i of the source's
// row is "in-edges before i dead, edge i live", of mass Q_{i-1} - Q_i in the
// gamma chain (total 2^62 - Q_d); z = floor(U (2^62 - Q_d) / 2^64) from the
// BUCKET-domain block of sample j picks the first edge e with
// 2^62 - Q_e > z, i.e. Q_e < 2^62 - z (the chain does not increase).
// Returns the edge position; the edges after it get FIRST coins of round 0.
template <bool kSeedKey = false>
__device__ __forceinline__ uint64_t bucket_pick(const SampleArgs& a, uint64_t j, uint64_t off, uint32_t deg) {
    const uint64_t one62 = 1ull << 62;
    const uint64_t G = one62 - a.chain[off + deg - 1];
    const uint4 x = kSeedKey ? coin_block(a.seed, 0, 0, kDomBucket, j) : coin_block(a.rk, 0, 0, kDomBucket, j);
    const uint64_t z = __umul64hi((uint64_t)x.x | ((uint64_t)x.y << 32), G);
    const uint64_t lim = one62 - z;
    uint32_t lo = 0, hi = deg - 1;  // the answer exists: Q_d = 2^62 - G < lim
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a.chain[off + mid] < lim) hi = mid;
        else lo = mid + 1;
    }
    return off + lo;
}

// The source record (source, in-row) of sample j, from the prepass when it
// holds j, else drawn; *pe receives the prepass's bucket pick (or -1).
__device__ __forceinline__ uint32_t source_of(const SampleArgs& a, uint64_t j, RowInfo* rv, int64_t* pe) {
    *pe = -1;
    if (a.up_rec && j - a.up_first < a.up_count) {
        const uint64_t t = j - a.up_first;
        const uint4 r = __ldg(a.up_rec + t);
        rv->deg = r.y;
        rv->off = r.z;
        rv->tau = r.w;
        if (a.up_pick && a.chain && r.y > 0) *pe = __ldg(&a.up_pick[t].x);
        return r.x;
    }
    const uint32_t v = draw_source(a, j);
    *rv = a.rows[v];
    return v;
}

// ----------------------------------------------------------- inserters
// Warp tier: the members of the warp's sample (which are also its BFS queue)
// and their hash set. Up to kQCap members live in shared memory; a larger
// sample moves both to the warp's spill slot in global memory (L2) and goes
// on there, up to spill.cap members. A candidate's in-row is loaded while its
// hash slot is probed, and kept in a shared ring if it joins within kRing
// places of the queue's head, so that a pop finds the row without going
// through the queue and the row table (a chain of two memory latencies per
// BFS level).
struct WarpInserter {
    uint32_t* hash;
    int32_t* queue;
    uint4* ring;      // (offset, degree, threshold, queue position) of queued members
    uint32_t* ghash;  // the spill slot
    int32_t* gqueue;
    const RowInfo* rows;
    SpillSize spill;
    uint32_t qlen, head;
    bool big;         // the sample lives in the spill slot
    bool overflow;

    // u joins table h (mask + 1 slots); false if it is there already
    static __device__ __forceinline__ bool put(uint32_t* table, uint32_t h, uint32_t mask, uint32_t u) {
        for (;;) {
            const uint32_t old = atomicCAS(&table[h], kEmpty, u);
            if (old == kEmpty) return true;
            if (old == u) return false;
            h = (h + 1) & mask;
        }
    }

    __device__ __forceinline__ bool put_shared(uint32_t u) {
        return put(hash, (u * 2654435761u) >> (32 - kHashBits), kHCap - 1, u);
    }
    __device__ __forceinline__ bool put_spill(uint32_t u) {
        return put(ghash, (u * 2654435761u) >> (32 - spill.hash_bits), (1u << spill.hash_bits) - 1, u);
    }

    // The sample outgrew shared memory: its members (qlen of them, and the
    // lanes' fresh ones) go to the spill slot, whose table is cleared first.
    __device__ __forceinline__ void move(int32_t u, bool fresh) {
        const int lane = threadIdx.x & 31;
        for (uint32_t i = lane; i < (1u << spill.hash_bits) / 4; i += 32)
            reinterpret_cast<uint4*>(ghash)[i] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
        __syncwarp();
        for (uint32_t i = lane; i < qlen; i += 32) {
            const int32_t w = queue[i];
            gqueue[i] = w;
            put_spill((uint32_t)w);
        }
        if (fresh) put_spill((uint32_t)u);
        big = true;
        __syncwarp();
    }

    __device__ __forceinline__ void insert(int32_t u) {
        if (overflow) return;  // warp-uniform
        bool fresh = false;
        uint4 rw = make_uint4(0, 0, 0, 0);  // the row record's words: offset (low, high), degree, threshold
        if (u >= 0) {
            rw = __ldg(reinterpret_cast<const uint4*>(rows) + u);  // in flight while the table is probed
            fresh = big ? put_spill((uint32_t)u) : put_shared((uint32_t)u);
        }
        const unsigned m = __ballot_sync(kFull, fresh);
        if (m) {
            const uint32_t pos = qlen + __popc(m & lanemask_lt());
            const uint32_t len = qlen + __popc(m);
            if (len > (uint32_t)kQCap && !big) move(u, fresh);
            if (len > spill.cap) {
                overflow = true;
            } else if (fresh) {
                if (big) gqueue[pos] = u;
                else queue[pos] = u;
                if (pos - head < (uint32_t)kRing) ring[pos & (kRing - 1)] = make_uint4(rw.x, rw.z, rw.w, pos);
            }
            qlen = len;
        }
        __syncwarp();
    }

    __device__ __forceinline__ int32_t member(uint32_t i) const { return big ? gqueue[i] : queue[i]; }
};

__device__ __forceinline__ uint32_t min4(const uint4& x) { return min(min(x.x, x.y), min(x.z, x.w)); }

__device__ __forceinline__ uint32_t min8(const uint4& x, const uint4& y) {
    return __vimin3_u32(__vimin3_u32(x.x, x.y, x.z), __vimin3_u32(x.w, y.x, y.y), min(y.z, y.w));
}

// Live mask of edge quad q (block x, thresholds t; bit k: edge 4 q + k) within
// its row's edges [lo, hi).
__device__ __forceinline__ unsigned quad_live(uint32_t q, const uint4& x, const uint4& t, uint32_t lo, uint32_t hi) {
    const uint32_t e0 = q << 2;
    const unsigned live = (coin_live(x.x, t.x) ? 1u : 0u) | (coin_live(x.y, t.y) ? 2u : 0u) |
                          (coin_live(x.z, t.z) ? 4u : 0u) | (coin_live(x.w, t.w) ? 8u : 0u);
    const uint32_t before = e0 < lo ? lo - e0 : 0u, after = e0 + 4 > hi ? e0 + 4 - hi : 0u;
    return live & (15u << before) & (15u >> after);
}

__device__ __forceinline__ uint32_t row_quads(uint32_t lo, uint32_t hi) {
    return hi > lo ? ((hi - 1) >> 2) - (lo >> 2) + 1 : 0u;
}

// The rejection form's accepted round for a source row of 1 to 16 edge quads,
// by one warp: rounds are independent given (j, r), so 32 / nq of them are
// drawn a pass, lane g taking quad g % nq of round r + g / nq, and the first
// lane with a live coin is in the accepted round, as in sequential order.
// Returns the cap when no round below it is accepted.
__device__ __forceinline__ uint32_t accepted_round(const SampleArgs& a, uint64_t j, uint32_t lo, uint32_t hi,
                                                   uint32_t tau) {
    const int lane = threadIdx.x & 31;
    const uint32_t nq = row_quads(lo, hi), rounds = 32u / nq, ri = (uint32_t)lane / nq;
    const uint32_t q = (lo >> 2) + (uint32_t)lane % nq;
    const uint4 t4 = a.tau ? __ldg(reinterpret_cast<const uint4*>(a.tau) + q) : make_uint4(tau, tau, tau, tau);
    for (uint32_t r = 0; r < a.retry_cap; r += rounds) {
        unsigned live = 0;
        if (ri < rounds && r + ri < a.retry_cap)
            live = quad_live(q, coin_block(a.rk, q, r + ri, kDomFirst, j), t4, lo, hi);
        const unsigned bal = __ballot_sync(kFull, live != 0u);
        if (bal) return r + (uint32_t)(__ffs(bal) - 1) / nq;
    }
    return a.retry_cap;
}
constexpr uint32_t kShortRow = 16;  // longest source row (edge quads) whose rounds are searched by accepted_round

// The edge quads of up to 32 rows laid end to end, two a lane and step: the
// rows with edges are packed into shared memory (first quad, first and end
// edge, threshold), and the row of quad g is the number of rows that start at
// or before it, a popcount of the step's row starts (one OR-reduction of the
// rows' start bits).
struct RowBatch {
    uint4* row;       // the warp's 32 packed rows
    uint32_t nq, excl, total;

    // lane's row: edges [lo, hi), threshold tau; nq edge quads of it are drawn (0: none)
    __device__ __forceinline__ RowBatch(uint4* rows, uint32_t lo, uint32_t hi, uint32_t tau, uint32_t nq_)
        : row(rows), nq(nq_) {
        const int lane = threadIdx.x & 31;
        uint32_t incl = nq;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += y;
        }
        total = __shfl_sync(kFull, incl, 31);
        excl = incl - nq;
        const unsigned m = __ballot_sync(kFull, nq > 0);
        __syncwarp();  // the last batch's rows are read (shuffles and votes order no memory)
        if (nq) row[__popc(m & lanemask_lt())] = make_uint4(excl, lo, hi, tau);
        __syncwarp();
    }

    // rows that start before quad `base`
    __device__ __forceinline__ uint32_t started(uint32_t base) const {
        return (uint32_t)__popc(__ballot_sync(kFull, nq && excl < base));
    }

    // the packed row of quad base + lane, *st rows starting before base (advanced past the 32 quads);
    // past the batch's end the last row
    __device__ __forceinline__ uint4 find(uint32_t base, uint32_t* st) const {
        const uint32_t d = excl - base;
        const unsigned m = __reduce_or_sync(kFull, nq && d < 32u ? 1u << d : 0u);
        const uint32_t i = *st + __popc(m & (lanemask_lt() | (1u << (threadIdx.x & 31)))) - 1;
        *st += __popc(m);
        return row[i];
    }

    // Draws the BFS coins of quads [base, base + 64) of sample blk and hands
    // each lane's live masks to list(quad, mask) (called warp-uniformly, with no lanes missing).
    template <class List>
    __device__ __forceinline__ void step(const SampleArgs& a, const SampleBlock& blk, uint32_t base, uint32_t* st,
                                         List&& list) const {
        const uint4* __restrict__ tau4 = reinterpret_cast<const uint4*>(a.tau);
        const uint32_t g0 = base + (threadIdx.x & 31), g1 = g0 + 32;
        const uint4 r0 = find(base, st), r1 = find(base + 32, st);
        // lanes past the batch's end take its last quad and drop its coins
        const uint32_t q0 = (r0.y >> 2) + (min(g0, total - 1) - r0.x);
        const uint32_t q1 = (r1.y >> 2) + (min(g1, total - 1) - r1.x);
        const bool two = base + 32 < total;  // warp-uniform
        const uint4 t0 = tau4 ? __ldg(tau4 + q0) : make_uint4(r0.w, r0.w, r0.w, r0.w);
        unsigned l0 = 0, l1 = 0;
        if (two) {  // two independent blocks
            const uint4 t1 = tau4 ? __ldg(tau4 + q1) : make_uint4(r1.w, r1.w, r1.w, r1.w);
            const uint4 x0 = blk(q0, a.rk), x1 = blk(q1, a.rk);
            l0 = quad_live(q0, x0, t0, r0.y, r0.z);
            if (g1 < total) l1 = quad_live(q1, x1, t1, r1.y, r1.z);
        } else if (g0 < total) {
            l0 = quad_live(q0, blk(q0, a.rk), t0, r0.y, r0.z);
        }
#pragma unroll 1
        for (int h = 0; h < (two ? 2 : 1); ++h) list(h ? q1 : q0, h ? l1 : l0);
    }
};

// The live edges (mask of edge quad q) of every lane join the warp's list of
// edge positions; returns the list's new length (at most 128 more).
__device__ __forceinline__ uint32_t list_live(uint32_t* pend, uint32_t npend, uint32_t q, unsigned live) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned m = __ballot_sync(kFull, (live >> k) & 1u);
        if ((live >> k) & 1u) pend[npend + __popc(m & lanemask_lt())] = 4u * q + (uint32_t)k;
        npend += __popc(m);
    }
    return npend;
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(kFull, v, d);
    return __shfl_sync(kFull, v, 0);
}

__device__ __forceinline__ void record_retry_failure(const SampleArgs& a, uint64_t j, uint32_t v, uint32_t r,
                                                     uint32_t deg) {
    a.h_off[j - a.id_base] = 0;
    a.h_len[j - a.id_base] = 0;
    a.h_src[j - a.id_base] = v;
    a.h_retries[j - a.id_base] = r;
    a.h_coins[j - a.id_base] = (uint64_t)deg * r;
    atomicOr(&a.status->flags, kStRetry);
    atomicMin(&a.status->first_bad, (unsigned long long)j);
}

// Alg. 1's source draw for every input id at once: the source of sample j and its
// in-row, as 16 bytes (source, degree, row offset, row threshold), so that a
// lane-tier lane starting a sample makes one coalesced load; with the bucket
// form, also the first step's picked in-edge and its source (8 bytes), whose
// dependent chain loads are better spread over this many-thread pass than
// paid by a lane at claim time. Row offsets fit 32 bits because graphs hold
// fewer than 2^32 - 8 edges.
__global__ void k_sources(SampleArgs a, uint4* __restrict__ rec, uint2* __restrict__ pick) {
    const uint64_t count = input_count(a);
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t j = input_id(a, t);
        const uint32_t v = draw_source<true>(a, j);
        const RowInfo rv = a.rows[v];
        rec[t] = make_uint4(v, rv.deg, (uint32_t)rv.off, rv.tau);
        if (a.chain && rv.deg > 0) {  // the bucket form of the first step, drawn here in bulk
            const uint64_t e = bucket_pick<true>(a, j, rv.off, rv.deg);
            pick[t] = make_uint2((uint32_t)e, (uint32_t)a.src[e]);
        }
    }
}

__device__ __forceinline__ uint64_t shfl_u64(uint64_t v, int src) {
    const uint32_t lo = __shfl_sync(kFull, (uint32_t)v, src);
    const uint32_t hi = __shfl_sync(kFull, (uint32_t)(v >> 32), src);
    return ((uint64_t)hi << 32) | lo;
}

// ------------------------------------------------------------- lane tier
// One lane per sample with a lean inner step: one edge quad of the lane's
// current row (Philox block, thresholds, four compares); live coins join the
// member list at once (visited check by scanning it); at the end of a row
// the next queued member's row, loaded ahead, takes over. Finished samples
// are written out, and idle lanes refilled, in batches: when at least
// kLaneRefill lanes are idle or nothing else is left.
constexpr int kLaneBlock = 256;
constexpr int kLaneQ = 32;
constexpr int kLaneStride = kLaneQ + 1;  // odd: conflict-free by lane and by member
constexpr int kLaneRefill = 8;

// One of 64 bits for vertex u (the top six bits of a multiplicative hash): a
// lane's sample keeps the OR over its members, so a candidate whose bit is
// clear is new without searching the member list.
__device__ __forceinline__ uint64_t member_bit(uint32_t u) { return 1ull << ((u * 0x9E3779B9u) >> 26); }

__global__ void __launch_bounds__(kLaneBlock, 4) k_iis_lane(SampleArgs a) {
    __shared__ int32_t s_q[kLaneBlock / 32][32 * kLaneStride];
    const int lane = threadIdx.x & 31;
    int32_t* const mq = s_q[threadIdx.x >> 5];
    int32_t* const mine = mq + lane * kLaneStride;
    const uint64_t count = input_count(a);
    const uint4* __restrict__ tau4 = reinterpret_cast<const uint4*>(a.tau);
    const int4* __restrict__ src4 = reinterpret_cast<const int4*>(a.src);

    bool busy = false, done = false, first = false, any = false, pf_ok = false;
    uint64_t j = 0, coins = 0;
    uint32_t v = 0, r = 0, len = 0, head = 0, src_deg = 0, tau_row = 0, steps = 0;
    uint32_t lo = 0, hi = 0, qc = 0, q_last = 0;
    uint32_t pf_off = 0, pf_deg = 0, pf_tau = 0;
    bool exhausted = false;
    uint64_t pool_base = 0;
    uint32_t pool_n = 0, pool_used = 0;
    uint4 rec = make_uint4(0, 0, 0, 0);
    uint2 prec = make_uint2(0, 0);
    uint64_t sig = 0;  // the sample's members, one hashed bit each (member_bit)
    uint64_t chunk_pos = 0, chunk_end = 0;
    uint32_t chunk = kLaneArenaChunk;

    for (;;) {
        // ---- batched maintenance: write out finished samples, refill
        const unsigned dn = __ballot_sync(kFull, done);
        const unsigned free_l = __ballot_sync(kFull, !busy || done);
        const bool all_free = free_l == kFull;
        if (__popc(free_l) >= kLaneRefill || all_free) {
            if (dn) {
                const uint32_t mylen = done ? len : 0u;
                uint32_t incl = mylen;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += y;
                }
                const uint32_t total = __shfl_sync(kFull, incl, 31);
                bool fits = true;
                if (chunk_end - chunk_pos < total) {
                    const uint64_t size = max((uint64_t)chunk, (uint64_t)total);
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(a.arena_cursor, (unsigned long long)size);
                    base = __shfl_sync(kFull, base, 0);
                    if (base + size > a.arena_cap) {
                        fits = false;
                        chunk = 0;
                        chunk_pos = chunk_end = 0;
                    } else {
                        chunk_pos = base;
                        chunk_end = base + size;
                    }
                }
                const uint64_t at = chunk_pos + (incl - mylen);
                if (done) {
                    if (fits) {
                        a.h_off[j - a.id_base] = at;
                        a.h_len[j - a.id_base] = len;
                        a.h_src[j - a.id_base] = v;
                        a.h_retries[j - a.id_base] = r;
                        a.h_coins[j - a.id_base] = coins;
                    } else {
                        arena_overflow(a, j);
                    }
                }
                __syncwarp();
                if (fits && total < 16u * (uint32_t)__popc(dn)) {
                    // short samples: their members end to end over the warp's
                    // lanes, each lane finding the sample that holds its entry
                    // (the first lane whose inclusive end exceeds it)
                    const uint32_t excl = incl - mylen;
                    for (uint32_t b0 = 0; b0 < total; b0 += 32) {
                        const uint32_t idx = b0 + (uint32_t)lane;
                        int owner = 0;
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1)
                            if (__shfl_sync(kFull, incl, owner + step - 1) <= idx) owner += step;
                        const uint32_t start = __shfl_sync(kFull, excl, owner);
                        if (idx < total) {
                            const int32_t u = mq[owner * kLaneStride + (idx - start)];
                            a.arena[chunk_pos + idx] = u;
                            count_member(a, u);
                        }
                    }
                    chunk_pos += total;
                } else if (fits) {
                    unsigned m = dn;
                    while (m) {
                        const int sl = __ffs(m) - 1;
                        m &= m - 1;
                        const uint64_t at_s = shfl_u64(at, sl);
                        const uint32_t len_s = __shfl_sync(kFull, len, sl);
                        if ((uint32_t)lane < len_s) {
                            const int32_t u = mq[sl * kLaneStride + lane];
                            a.arena[at_s + lane] = u;
                            count_member(a, u);
                        }
                    }
                    chunk_pos += total;
                }
                __syncwarp();
                if (done) {
                    done = false;
                    busy = false;
                }
            }
            unsigned idle = __ballot_sync(kFull, !busy);
            while (idle && !exhausted) {
                if (pool_used == pool_n) {
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(a.work, 32ull);
                    base = __shfl_sync(kFull, base, 0);
                    if (base >= count) {
                        exhausted = true;
                        break;
                    }
                    pool_base = base;
                    pool_n = (uint32_t)min(32ull, count - base);
                    pool_used = 0;
                    if ((uint32_t)lane < pool_n) {
                        rec = __ldg(a.srcrec + base + lane);
                        if (a.srcpick) prec = __ldg(a.srcpick + base + lane);
                    }
                }
                const uint32_t take = min((uint32_t)__popc(idle), pool_n - pool_used);
                const uint32_t rank = __popc(idle & lanemask_lt());
                const int from = (int)min(pool_used + rank, 31u);
                const uint32_t rv_src = __shfl_sync(kFull, rec.x, from);
                const uint32_t rv_deg = __shfl_sync(kFull, rec.y, from);
                const uint32_t rv_off = __shfl_sync(kFull, rec.z, from);
                const uint32_t rv_tau = __shfl_sync(kFull, rec.w, from);
                const uint32_t pk_e = __shfl_sync(kFull, prec.x, from);
                const uint32_t pk_u = __shfl_sync(kFull, prec.y, from);
                if (!busy && rank < take) {
                    j = input_id(a, pool_base + pool_used + rank);
                    v = rv_src;  // Alg. 1's source, drawn by k_sources
                    if (rv_deg > a.max_deg) {
                        hand_on(a, j);
                    } else {
                        busy = true;
                        first = true;
                        any = false;
                        pf_ok = false;
                        r = 0;
                        mine[0] = (int32_t)v;
                        sig = member_bit(v);
                        len = 1;
                        head = 1;
                        src_deg = rv_deg;
                        tau_row = rv_tau;
                        lo = rv_off;
                        hi = rv_off + rv_deg;
                        q_last = hi > lo ? (hi - 1) >> 2 : lo >> 2;
                        if (a.srcpick) {  // bucket form: the picked in-edge, round-0 coins after it
                            mine[1] = (int32_t)pk_u;
                            sig |= member_bit(pk_u);
                            len = 2;
                            lo = pk_e + 1;
                            any = true;
                        }
                        qc = lo >> 2;
                        coins = 0;
                        steps = 0;
                    }
                }
                pool_used += take;
                idle = __ballot_sync(kFull, !busy);
            }
            if (!__any_sync(kFull, busy)) {
                if (exhausted) break;
                continue;
            }
        }
        if (!busy || done) continue;  // the lane waits for the next batch

        // ---- one edge quad: coins of the first step (round r) or of the
        // reverse BFS; a RIS source may have no in-edges
        bool handed = false, failed = false;
        uint32_t qdone = qc;  // the last quad drawn in this step
        if (hi > lo) {
            // up to two quads of the row per step: their thresholds, sources
            // and Philox blocks are independent, so their latencies overlap
            const bool two = qc < q_last;
            qdone = two ? qc + 1 : qc;
            const uint4 t4 = a.tau ? __ldg(tau4 + qc) : make_uint4(tau_row, tau_row, tau_row, tau_row);
            const uint4 t4b = (two && a.tau) ? __ldg(tau4 + qc + 1) : make_uint4(tau_row, tau_row, tau_row, tau_row);
            const uint32_t rr = first ? r : 0u, dom = first ? kDomFirst : kDomBfs;
            const uint4 x = coin_block(a.rk, qc, rr, dom, j);
            uint4 xb = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
            if (two) xb = coin_block(a.rk, qc + 1, rr, dom, j);
            const uint32_t e0 = qc << 2, e1 = e0 + 4;
            unsigned live = 0;
            live |= (e0 + 0 >= lo && e0 + 0 < hi && coin_live(x.x, t4.x)) ? 1u : 0u;
            live |= (e0 + 1 >= lo && e0 + 1 < hi && coin_live(x.y, t4.y)) ? 2u : 0u;
            live |= (e0 + 2 >= lo && e0 + 2 < hi && coin_live(x.z, t4.z)) ? 4u : 0u;
            live |= (e0 + 3 >= lo && e0 + 3 < hi && coin_live(x.w, t4.w)) ? 8u : 0u;
            if (two) {  // e1 > lo: only the row's end bounds the second quad
                live |= (e1 + 0 < hi && coin_live(xb.x, t4b.x)) ? 16u : 0u;
                live |= (e1 + 1 < hi && coin_live(xb.y, t4b.y)) ? 32u : 0u;
                live |= (e1 + 2 < hi && coin_live(xb.z, t4b.z)) ? 64u : 0u;
                live |= (e1 + 3 < hi && coin_live(xb.w, t4b.w)) ? 128u : 0u;
            }
            if (live) {
                any = true;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const unsigned lh = (live >> (4 * h)) & 15u;
                    if (!lh || handed) continue;
                    const int4 s4 = __ldg(src4 + qc + h);
                    const int32_t cand[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (!((lh >> k) & 1u) || handed) continue;
                        const int32_t u = cand[k];
                        bool seen = false;
                        if (sig & member_bit(u))  // else u is certainly new
                            for (uint32_t i = 0; i < len; ++i)
                                if (mine[i] == u) { seen = true; break; }
                        if (seen) continue;
                        if (len == (uint32_t)kLaneQ) handed = true;  // the warp tier takes it
                        else {
                            mine[len++] = u;
                            sig |= member_bit(u);
                        }
                    }
                }
            }
            steps += two ? 2u : 1u;
        }
        if (!handed && (hi <= lo || qdone >= q_last)) {  // the row is used up
            if (first) {
                if (any || a.ris) {
                    first = false;
                    coins = (uint64_t)src_deg * (r + 1);
                } else if (++r >= a.retry_cap) {
                    failed = true;
                } else if (r >= a.max_retries) {
                    handed = true;  // a rare source: the warp tier searches rounds in parallel
                } else {
                    qc = lo >> 2;  // next round over the same row
                }
            }
            if (!first && !failed && !handed) {
                // Alg. 1's reverse BFS: pop the next queued members until one
                // has in-edges (the first one's row was loaded ahead)
                bool row = false;
                while (!row && head < len) {
                    if (!pf_ok) {
                        const RowInfo rw = a.rows[mine[head]];
                        pf_off = (uint32_t)rw.off;
                        pf_deg = rw.deg;
                        pf_tau = rw.tau;
                    }
                    pf_ok = false;
                    ++head;
                    coins += pf_deg;
                    if (pf_deg > a.max_deg) {
                        handed = true;
                        break;
                    }
                    if (pf_deg > 0) {
                        row = true;
                        lo = pf_off;
                        hi = pf_off + pf_deg;
                        tau_row = pf_tau;
                        qc = lo >> 2;
                        q_last = (hi - 1) >> 2;
                    }
                }
                if (!row && !handed) done = true;
            }
        } else if (!handed) {
            qc = qdone + 1;
        }
        if (!done && !handed && steps > a.max_steps) handed = true;
        if (handed) hand_on(a, j);
        if (failed) record_retry_failure(a, j, v, r, src_deg);
        if (handed || failed) busy = false;
        // load the next pop's row ahead while this row's last quads are drawn
        if (busy && !done && !first && !pf_ok && head < len && q_last - qc <= 2u) {
            const RowInfo rw = a.rows[mine[head]];
            pf_off = (uint32_t)rw.off;
            pf_deg = rw.deg;
            pf_tau = rw.tau;
            pf_ok = true;
        }
    }
}

// ------------------------------------------------------------- warp tier
// One warp per sample. Up to 32 queued rows are taken at a time and their edge
// quads dealt to the lanes (RowBatch). Live edges are only listed (their
// positions, in shared memory) and joined 32 at a time, one a lane, so that
// the source gather, the probe and the row load of 32 candidates overlap and
// an insert round has every lane busy.
// Two thirds of a weighted-cascade sketch's members lie in samples of more
// than 256 members, so the tier goes on past shared memory. On 1M samples of
// Chung-Lu 1M / 17.5M WC this tier and the CTA tier took 29 ms when samples
// left here at 256 members and 7.5 ms now.
__global__ void __launch_bounds__(kWarpThreads, 4) k_iis_warp(SampleArgs a) {
    __shared__ __align__(16) uint32_t s_hash[kWarpThreads / 32][kHCap];
    __shared__ __align__(16) int32_t s_queue[kWarpThreads / 32][kQCap];
    __shared__ uint4 s_ring[kWarpThreads / 32][kRing];
    __shared__ uint4 s_row[kWarpThreads / 32][32];
    __shared__ uint32_t s_pend[kWarpThreads / 32][kPend];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint64_t wid = (uint64_t)blockIdx.x * (kWarpThreads / 32) + wib;
    uint32_t* const hash = s_hash[wib];
    uint32_t* const pend = s_pend[wib];
    uint64_t chunk_pos = 0, chunk_end = 0;  // this warp's arena reservation
    uint32_t chunk = kArenaChunk;

    const uint64_t count = input_count(a);
    // ids per cursor atomic: one where samples are few, so that every warp has
    // some (their costs differ a thousandfold), up to kIdBatch where they are many
    const uint64_t nwarps = (uint64_t)gridDim.x * (kWarpThreads / 32);
    const uint64_t batch = max((uint64_t)1, min((uint64_t)kIdBatch, count / (8 * nwarps)));
    for (;;) {
        unsigned long long t0 = 0;
        if (lane == 0) t0 = atomicAdd(a.work, (unsigned long long)batch);
        t0 = __shfl_sync(kFull, t0, 0);
        if (t0 >= count) break;
        const uint64_t t1 = min((uint64_t)t0 + batch, count);
        for (uint64_t t = t0; t < t1; ++t) {
            const uint64_t j = input_id(a, t);
            // clear the visited set and the ring
#pragma unroll
            for (int i = lane; i < kHCap / 4; i += 32)
                reinterpret_cast<uint4*>(hash)[i] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
#pragma unroll
            for (int i = lane; i < kRing; i += 32) s_ring[wib][i].w = kEmpty;
            __syncwarp();

            // Alg. 1: the source, alone in the sample
            RowInfo rv;
            int64_t pe;
            const uint32_t v = source_of(a, j, &rv, &pe);
            WarpInserter ins{hash, s_queue[wib], s_ring[wib], a.spill_hash + (wid << a.spill.hash_bits),
                             a.spill_queue + wid * a.spill.cap, a.rows, a.spill, 1u, 1u, false, false};
            if (lane == 0) {
                ins.put_shared(v);
                s_queue[wib][0] = (int32_t)v;
            }
            __syncwarp();

            uint32_t npend = 0;
            // the sources of the last cnt listed edges join the sample, one a lane
            auto join = [&](uint32_t cnt) {
                __syncwarp();
                npend -= cnt;
                const int32_t u = (uint32_t)lane < cnt ? __ldg(a.src + pend[npend + lane]) : -1;
                ins.insert(u);
            };
            auto list = [&](uint32_t q, unsigned live) {
                if (!__any_sync(kFull, live != 0u)) return;
                npend = list_live(pend, npend, q, live);
#pragma unroll 1
                while (npend >= 32u) join(32u);
            };
            // the FIRST coins of round r on the source's in-edges [lo, hi); whether one is live
            auto first_row = [&](uint32_t lo, uint32_t hi, uint32_t r) -> bool {
                const uint32_t qe = (lo >> 2) + row_quads(lo, hi);
                bool any = false;
#pragma unroll 1
                for (uint32_t qb = lo >> 2; qb < qe && !ins.overflow; qb += 32) {
                    const uint32_t q = qb + lane;
                    unsigned live = 0;
                    if (q < qe) {
                        const uint4 t4 = a.tau ? __ldg(reinterpret_cast<const uint4*>(a.tau) + q)
                                               : make_uint4(rv.tau, rv.tau, rv.tau, rv.tau);
                        live = quad_live(q, coin_block(a.rk, q, r, kDomFirst, j), t4, lo, hi);
                    }
                    any |= live != 0u;
                    list(q, live);
                }
                return __any_sync(kFull, any);
            };

            // Alg. 1's conditioned first step: the bucket form's picked in-edge
            // and round-0 coins after it, RIS's one round whatever its coins, or
            // the first round with a live coin
            const uint32_t s_lo = (uint32_t)rv.off, s_hi = s_lo + rv.deg;
            uint32_t r = 0, from = s_lo;
            if (a.chain) {
                uint32_t e = 0;
                if (lane == 0) {
                    e = pe >= 0 ? (uint32_t)pe : (uint32_t)bucket_pick(a, j, rv.off, rv.deg);
                    pend[0] = e;
                }
                npend = 1;
                from = __shfl_sync(kFull, e, 0) + 1;
            } else if (!a.ris && row_quads(s_lo, s_hi) <= kShortRow) {
                r = accepted_round(a, j, s_lo, s_hi, rv.tau);
            }
            bool failed = r >= a.retry_cap;
            while (!failed && !first_row(from, s_hi, r) && !a.chain && !a.ris) failed = ++r >= a.retry_cap;
            if (failed) {
                if (lane == 0) record_retry_failure(a, j, v, r, rv.deg);
                __syncwarp();
                continue;
            }

            // reverse BFS over the queue, up to 32 vertices at a time
            uint64_t coins = lane == 0 ? (uint64_t)rv.deg * (r + 1) : 0;
            uint64_t drawn = 0;  // in-edges of the rows taken so far (warp-uniform)
            bool heavy = false;
            const SampleBlock blk(a.rk, j, kDomBfs);
            for (;;) {
                if (ins.head >= ins.qlen && npend) join(npend);  // the level's last live edges (under 32)
                if (ins.head >= ins.qlen || ins.overflow) break;
                const uint32_t cnt = min(ins.qlen - ins.head, 32u);
                uint32_t lo = 0, deg = 0, tau_row = 0;
                if ((uint32_t)lane < cnt) {
                    const uint32_t pos = ins.head + lane;
                    const uint4 c = s_ring[wib][pos & (kRing - 1)];
                    if (c.w == pos) {
                        lo = c.x;
                        deg = c.y;
                        tau_row = c.z;
                    } else {  // it joined too far from the head for the ring
                        const RowInfo rw = a.rows[ins.member(pos)];
                        lo = (uint32_t)rw.off;
                        deg = rw.deg;
                        tau_row = rw.tau;
                    }
                }
                ins.head += cnt;
                // a sample that reaches huge in-rows goes to the CTA tier,
                // where every warp of a block shares its rows
                drawn += __reduce_add_sync(kFull, min(deg, 1u << 26));
                if (drawn > a.warp_max_coins) {
                    heavy = true;
                    break;
                }
                coins += deg;
                const RowBatch rb(s_row[wib], lo, lo + deg, tau_row, row_quads(lo, lo + deg));
                uint32_t st = 0;
#pragma unroll 1
                for (uint32_t base = 0; base < rb.total && !ins.overflow; base += 64) rb.step(a, blk, base, &st, list);
            }
            if (ins.overflow || heavy) {  // more members or coins than the tier takes: CTA tier
                if (lane == 0) hand_on(a, j);
                __syncwarp();
                continue;
            }
            coins = warp_sum_u64(coins);

            // arena append from this warp's chunk
            const uint32_t len = ins.qlen;
            if (chunk_end - chunk_pos < len) {
                const uint64_t size = max((uint64_t)chunk, (uint64_t)len);
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(a.arena_cursor, (unsigned long long)size);
                base = __shfl_sync(kFull, base, 0);
                if (base + size > a.arena_cap) {
                    chunk = 0;
                    chunk_pos = chunk_end = 0;
                    if (lane == 0) arena_overflow(a, j);
                    continue;
                }
                chunk_pos = base;
                chunk_end = base + size;
            }
            for (uint32_t i = lane; i < len; i += 32) {
                const int32_t u = ins.member(i);
                a.arena[chunk_pos + i] = u;
                count_member(a, u);
            }
            if (lane == 0) {
                a.h_off[j - a.id_base] = chunk_pos;
                a.h_len[j - a.id_base] = len;
                a.h_src[j - a.id_base] = v;
                a.h_retries[j - a.id_base] = r;
                a.h_coins[j - a.id_base] = coins;
            }
            chunk_pos += len;
            __syncwarp();
        }
    }
}

// -------------------------------------------------------------- CTA tier
// One block of kCtaThreads threads per sample, 1024 threads of such blocks per
// SM: eight blocks of 128 by default, or four of 256 or two of 512 where
// SKIS_OPT_CTA_THREADS asks for them.
// Four warps a sample pay a level's fixed cost half as often as eight, and
// twice as many samples hide one another's latencies. R-MAT 2^22 / 2^27 WC,
// 200K samples: 47.2 ms with blocks of 256, 44.7 with 128, 48.0 with 64;
// 2^25 / 2^30, 10^6 samples: 614, 600, 607; Chung-Lu 4M / 140M WC, 262K
// samples: 4.2, 2.9, 2.8.
// The reverse BFS goes level by level. The in-rows of a level's first
// kCtaWin vertices wait in shared memory: a vertex's row is loaded while its
// visited bit is set, so a level costs two memory latencies (the source
// gather, then the bit with the row) and one block barrier. Weighted cascade
// has narrow levels, a few rows each, and is bound by these.
// A level's rows go to the warps 32 at a time, a batch split over several
// warps where there are fewer batches than warps (RowBatch); rows of
// cta_hub_quads edge quads or more are strided over the whole block. Live
// edges are listed per warp and joined 32 at a time, the rest at the end of
// the level. Before, each of a quad's four words was inserted in turn (four
// atomic round trips a level) and every level read its queue and rows back:
// on Chung-Lu 1M / 17.5M WC the 7670 samples of 1M that run here took 7.4 ms
// and take 4.4 ms. Where hubs hold the coins it is bound by the coin
// generator: R-MAT 2^22 / 2^27 WC 372G blocks/s, 2^25 / 2^30 431G (the hub
// loop alone, with no other work in the kernel, 455G).
// Where a good part of a pass comes here, hubs hold the coins; then few
// samples are bound by the longest of them, which a larger block shortens. Tier
// alone, ms, blocks of 512 / 256 / 128: R-MAT 2^22 / 2^27, every sample here,
// 1,200 samples 1.90 / 1.89 / 2.78, 5K 2.7 / 2.8 / 3.8, 10K 4.3 / 4.2 / 5.1,
// 20K 7.3 / 6.8 / 6.9; 2^20 / 2^25 .98 / .99 / 1.30, 1.62 / 1.69 / 1.99, 2.46 /
// 2.12 / 2.41, 4.2 / 3.5 / 3.4; 2^18 / 2^23 at 5K .91 / .77 / .97; the default
// split of 10K samples of 2^20 / 2^25 (26 % here) 2.33 / 2.13 / 2.50. Where
// only the largest come here (Chung-Lu 4M / 140M WC, 1.7 % of 65K: 2.5 / 1.56 /
// 1.24, of 1M: 30 / 15.3 / 10.1) their levels are narrow and more of them at a
// time count. So blocks of 128, but for passes of which more than 1 /
// kCtaHubShare comes here: 512 up to kCtaFew samples an SM in the pass, 256 up
// to kCtaMany of them here.
constexpr int kCtaBlock = 128;
constexpr uint64_t kCtaHubShare = 8, kCtaFew = 24, kCtaMany = 96;
constexpr int kCtaWin = 512;  // rows of a level in shared memory at a time

template <int kCtaThreads>
__global__ void __launch_bounds__(kCtaThreads, 1024 / kCtaThreads) k_iis_cta(SampleArgs a, uint64_t above,
                                                                            uint64_t upto, bool within) {
    constexpr int kWarps = kCtaThreads / 32;
    const uint64_t count = input_count(a);
    if ((count > above && count <= upto) != within) return;  // the other launch's
    __shared__ unsigned long long s_j;
    __shared__ unsigned long long s_coins;
    __shared__ unsigned long long s_base;
    __shared__ uint4 s_win[2][kCtaWin];      // rows of this level and the next: first and end edge, threshold
    __shared__ uint16_t s_hub[2][kCtaWin];   // those of them that the hub loop takes
    // the previous, this and the next level's joins: vertices, hubs among them
    // in the window, edge quads of the others and chunks of 64 quads of the hubs
    struct Level {
        uint32_t size, hubs, quads, chunks;
    };
    __shared__ __align__(16) Level s_lvl[3];
    __shared__ uint4 s_row[kWarps][32];
    __shared__ uint32_t s_pend[kWarps][kPend];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t* const pend = s_pend[wid];
    uint32_t* bitmap = a.bitmaps + (uint64_t)blockIdx.x * a.bitmap_words;
    int32_t* queue = a.queues + (uint64_t)blockIdx.x * a.queue_cap;
    const uint4* __restrict__ tau4 = reinterpret_cast<const uint4*>(a.tau);
    const uint4* __restrict__ rows4 = reinterpret_cast<const uint4*>(a.rows);  // offset (low, high), degree, threshold
    auto is_hub = [&](uint32_t nq) { return a.cta_hub_quads && nq >= a.cta_hub_quads; };
    bool clean = a.slot_clean[blockIdx.x] != 0;
    unsigned long long claim = 0;  // thread 0: the block's next input
    if (threadIdx.x == 0) claim = atomicAdd(a.work, 1ull);

    for (;;) {
        if (threadIdx.x == 0) {
            s_j = claim < count ? input_id(a, claim) : ~0ull;
            s_coins = 0;
            s_lvl[0] = s_lvl[1] = s_lvl[2] = Level{0, 0, 0, 0};
        }
        __syncthreads();
        const uint64_t j = s_j;
        if (j == ~0ull) break;
        if (threadIdx.x == 0) claim = atomicAdd(a.work, 1ull);  // arrives while this sample is drawn
        if (!clean) {  // the slot's first sample: its bitmap is cleared once, and kept clear by every sample
            for (uint64_t i = threadIdx.x; i < a.bitmap_words; i += kCtaThreads) bitmap[i] = 0;
            __syncthreads();
            if (threadIdx.x == 0) a.slot_clean[blockIdx.x] = 1;
            clean = true;
        }

        RowInfo rv;
        int64_t pe;
        const uint32_t v = source_of(a, j, &rv, &pe);
        if (threadIdx.x == 0) {
            bitmap[v >> 5] |= 1u << (v & 31);
            queue[0] = (int32_t)v;
        }
        __syncthreads();  // the source's bit is set before any other

        uint32_t tail = 1;     // members before this level's joins
        uint64_t coins = 0;    // in-edges of the members that this lane joined
        int cur = 0, nxt = 1;  // this level's joins, the next level's (zero)
        int buf = 0;           // half of s_win that this level's joins fill
        uint32_t npend = 0;
        // the sources of the last cnt listed edges join the sample, one a lane.
        // A vertex past the queue's capacity gets its bit back, so that the
        // bitmap always holds exactly the queued vertices (the counter still
        // counts it: the sample is then known to have outgrown the slot)
        auto join = [&](uint32_t cnt) {
            __syncwarp();
            npend -= cnt;
            int32_t u = 0;
            bool fresh = false;
            uint4 rw = make_uint4(0, 0, 0, 0);
            if ((uint32_t)lane < cnt) {
                u = __ldg(a.src + pend[npend + lane]);
                rw = __ldg(rows4 + u);  // in flight while the bit is set
                fresh = (atomicOr(&bitmap[(uint32_t)u >> 5], 1u << (u & 31)) & (1u << (u & 31))) == 0;
            }
            const unsigned m = __ballot_sync(kFull, fresh);
            if (m) {
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&s_lvl[cur].size, (uint32_t)__popc(m));
                at = __shfl_sync(kFull, at, 0) + __popc(m & lanemask_lt());
                const uint32_t nq = fresh ? row_quads(rw.x, rw.x + rw.z) : 0u;
                const uint32_t quads = __reduce_add_sync(kFull, is_hub(nq) ? 0u : nq);
                if (lane == 0) atomicAdd(&s_lvl[cur].quads, quads);
                if (fresh) {
                    coins += rw.z;
                    if (tail + at < a.queue_cap) queue[tail + at] = u;
                    else atomicAnd(&bitmap[(uint32_t)u >> 5], ~(1u << (u & 31)));
                    if (at < (uint32_t)kCtaWin) {
                        s_win[buf][at] = make_uint4(rw.x, rw.x + rw.z, rw.w, 0u);
                        if (is_hub(nq)) {
                            s_hub[buf][atomicAdd(&s_lvl[cur].hubs, 1u)] = (uint16_t)at;
                            atomicAdd(&s_lvl[cur].chunks, (nq + 63) / 64);
                        }
                    }
                }
            }
            __syncwarp();
        };
        auto list = [&](uint32_t q, unsigned live) {
            if (!__any_sync(kFull, live != 0u)) return;
            npend = list_live(pend, npend, q, live);
#pragma unroll 1
            while (npend >= 32u) join(32u);
        };

        // Alg. 1's conditioned first step: the source row is strided over the
        // block in whole quads (a short row's rounds are searched by every warp
        // for itself, and its accepted round drawn by the first)
        const uint32_t s_lo = (uint32_t)rv.off, s_hi = s_lo + rv.deg;
        uint32_t r = 0, from = s_lo;
        const bool short_row = !a.chain && !a.ris && row_quads(s_lo, s_hi) <= kShortRow;
        if (a.chain) {
            uint32_t e = 0;
            if (lane == 0) e = pe >= 0 ? (uint32_t)pe : (uint32_t)bucket_pick(a, j, rv.off, rv.deg);
            e = __shfl_sync(kFull, e, 0);
            if (wid == 0) {
                if (lane == 0) pend[0] = e;
                npend = 1;
            }
            from = e + 1;
        } else if (short_row) {
            r = accepted_round(a, j, s_lo, s_hi, rv.tau);
        }
        bool failed = r >= a.retry_cap;
        while (!failed) {
            const uint32_t qe = (from >> 2) + row_quads(from, s_hi);
            bool any = false;
#pragma unroll 1
            for (uint32_t qb = (from >> 2) + wid * 32; qb < qe; qb += kCtaThreads) {
                const uint32_t q = qb + lane;
                unsigned live = 0;
                if (q < qe) {
                    const uint4 t4 = tau4 ? __ldg(tau4 + q) : make_uint4(rv.tau, rv.tau, rv.tau, rv.tau);
                    live = quad_live(q, coin_block(a.rk, q, r, kDomFirst, j), t4, from, s_hi);
                }
                any |= live != 0u;
                list(q, live);
            }
            if (a.chain || a.ris || short_row || __syncthreads_or(any ? 1 : 0)) break;
            failed = ++r >= a.retry_cap;
        }
        if (failed) {
            if (threadIdx.x == 0) {
                record_retry_failure(a, j, v, r, rv.deg);
                bitmap[v >> 5] = 0;
            }
            __syncthreads();
            continue;
        }
        if (npend) join(npend);

        // reverse BFS, level by level
        const SampleBlock blk(a.rk, j, kDomBfs);
        for (;;) {
            __syncthreads();  // the last level's joins are in
            const Level lvl = s_lvl[cur];
            const uint32_t size = lvl.size, head = tail;
            tail += size;
            if (size == 0 || tail > a.queue_cap) break;  // done, or the sample outgrew the slot
            // the counters rotate: this level fills `nxt` (zero), and the one
            // after that, read by every thread before this barrier, is cleared
            const int spare = 3 - cur - nxt;
            cur = nxt;
            nxt = spare;
            if (threadIdx.x == 0) s_lvl[nxt] = Level{0, 0, 0, 0};
            const uint4* const win = s_win[buf];
            const uint16_t* const hubs = s_hub[buf];
            buf ^= 1;
#pragma unroll 1
            for (uint32_t w0 = 0; w0 < size; w0 += kCtaWin) {
                const uint32_t nw = min((uint32_t)kCtaWin, size - w0);
                uint32_t nhub = lvl.hubs, chunks = lvl.chunks;
                if (w0) {  // a wide level's later rows: loaded from the queue
                    __shared__ uint32_t s_whub[2];
                    __syncthreads();
                    if (threadIdx.x < 2) s_whub[threadIdx.x] = 0;
                    __syncthreads();
                    for (uint32_t i = threadIdx.x; i < nw; i += kCtaThreads) {
                        const uint4 rw = __ldg(rows4 + queue[head + w0 + i]);
                        const uint32_t nq = row_quads(rw.x, rw.x + rw.z);
                        s_win[buf ^ 1][i] = make_uint4(rw.x, rw.x + rw.z, rw.w, 0u);
                        if (is_hub(nq)) {
                            s_hub[buf ^ 1][atomicAdd(&s_whub[0], 1u)] = (uint16_t)i;
                            atomicAdd(&s_whub[1], (nq + 63) / 64);
                        }
                    }
                    __syncthreads();
                    nhub = s_whub[0];
                    chunks = s_whub[1];
                }
                // batches of 32 rows, each dealt to 2^sh warps while warps are left
                // over (a narrow level's few quads go to the first warps, the
                // others do not look at its rows)
                const int batches = (int)((nw + 31) / 32);
                const int sh = max(0, 31 - __clz(kWarps) - (batches > 1 ? 32 - __clz(batches - 1) : 0));
                const uint32_t part = (uint32_t)wid & ((1u << sh) - 1u);
#pragma unroll 1
                for (int b = 64u * part < lvl.quads ? wid >> sh : batches; b < batches; b += kWarps >> sh) {
                    const uint32_t i = 32u * b + lane;
                    uint4 w = make_uint4(0, 0, 0, 0);
                    if (i < nw) w = win[i];
                    uint32_t nq = row_quads(w.x, w.y);
                    if (is_hub(nq)) nq = 0;  // the hub loop takes it
                    const RowBatch rb(s_row[wid], w.x, w.y, w.z, nq);
#pragma unroll 1
                    for (uint32_t base = 64u * part; base < rb.total; base += 64u << sh) {
                        uint32_t st = rb.started(base);
                        rb.step(a, blk, base, &st, list);
                    }
                }
                // hub rows: their chunks of 64 quads laid end to end and cut into one
                // run a warp, so a warp goes straight down a row with no search,
                // two independent blocks a lane and step. For one threshold a row
                // (never the sentinel: a hub has many edges) a step is one compare
                // of the blocks' minimum, as a live coin is rare there (weighted
                // cascade expects one a row)
                const uint32_t per = (chunks + kWarps - 1) / kWarps, run0 = wid * per;
                const uint32_t run1 = run0 < chunks ? min(chunks, run0 + per) : 0u;
                uint32_t before = 0;  // chunks of the hubs before h
#pragma unroll 1
                for (uint32_t h = 0; h < nhub && before < run1; ++h) {
                    const uint4 w = win[hubs[h]];
                    const uint32_t lo = w.x, hi = w.y, tr = w.z, nq = row_quads(lo, hi), n = (nq + 63) / 64;
                    const uint32_t c0 = max(run0, before) - before, c1 = min(run1, before + n) - before;
                    const bool mine = run0 < before + n;
                    before += n;
                    if (!mine) continue;
                    uint32_t q = (lo >> 2) + 64 * c0 + lane;  // this lane's quads: q and q + 32
                    const uint32_t qe = (lo >> 2) + nq;
                    // the live coins of one step join the list (quads past the row's end dropped)
                    auto draw = [&]() {
                        const uint4 tr4 = make_uint4(tr, tr, tr, tr);
#pragma unroll 1
                        for (uint32_t k = 0; k < 64 && q - lane + k < qe; k += 32) {
                            const uint32_t qk = q + k;
                            const uint4 x = blk(qk, a.rk);
                            if (!tau4 && !__any_sync(kFull, min4(x) < tr)) continue;
                            unsigned live = 0;
                            if (qk < qe) live = quad_live(qk, x, tau4 ? __ldg(tau4 + qk) : tr4, lo, hi);
                            list(qk, live);
                        }
                        q += 64;
                    };
                    uint32_t full = max(c0, min(c1, nq / 64)) - c0;  // steps without a ragged end
#pragma unroll 1
                    while (full) {
                        if (!tau4) {
                            // nothing but blocks and the compare until a lane may have a
                            // live coin, whose step is then drawn again
                            bool hit;
                            do {
                                hit = __any_sync(kFull, min8(blk(q, a.rk), blk(q + 32, a.rk)) < tr);
                                q += 64;
                                --full;
                            } while (!hit && full);
                            if (!hit) break;
                            q -= 64;
                        } else {
                            --full;
                        }
                        draw();
                    }
                    if (c1 == n && nq % 64) draw();
                }
            }
            if (npend) join(npend);
        }
        const uint32_t len = tail;
        coins = warp_sum_u64(coins);
        if (lane == 0 && coins) atomicAdd(&s_coins, (unsigned long long)coins);
        __syncthreads();
        const bool outgrown = len > a.queue_cap;  // the queue kept its first queue_cap members only
        if (threadIdx.x == 0) {
            const unsigned long long base = outgrown ? 0ull : atomicAdd(a.arena_cursor, (unsigned long long)len);
            if (outgrown) {  // to the pass whose slots hold n-entry queues
                if (a.out_ids) hand_on(a, j);
                else atomicOr(&a.status->flags, kStListFull);
                s_base = ~0ull;
            } else if (base + len > a.arena_cap) {
                arena_overflow(a, j);
                s_base = ~0ull;
            } else {
                s_base = base;
                a.h_off[j - a.id_base] = base;
                a.h_len[j - a.id_base] = len;
                a.h_src[j - a.id_base] = v;
                a.h_retries[j - a.id_base] = r;
                a.h_coins[j - a.id_base] = (uint64_t)rv.deg * (r + 1) + s_coins;
            }
        }
        __syncthreads();
        const unsigned long long base = s_base;
        for (uint32_t i = threadIdx.x; i < min(len, a.queue_cap); i += kCtaThreads) {
            const int32_t u = queue[i];
            if (base != ~0ull) {
                a.arena[base + i] = u;
                count_member(a, u);
            }
            bitmap[(uint32_t)u >> 5] = 0;  // restore the all-zero bitmap
        }
        __syncthreads();
    }
}

// --------------------------------------------------------------- LT walks
// Linear Threshold samples (Sec. "Extensions to other diffusion models",
// LT): the source by Eq. probu with gamma_v = the row's weight sum, exactly
// one in-neighbour picked with probability w(u,v) / gamma_v, then the
// reverse walk of RIS for LT: from the last member x, one draw picks at most
// one in-edge of x (edge i when P_{i-1} <= y < P_i for the running weight
// sums P, none when y >= P_d); the walk ends when none is picked or the
// picked vertex is already in R_j. Step t of sample j draws the Philox block
// (q = t, domain LT, sample j): step 0 conditioned (64-bit U, y = floor(U S
// / 2^64)), later steps y = its word 0. Three tiers: a lane a walk with up to
// kLtQ members in shared memory, a lane a walk with up to kLtMidCap members in
// global memory, then one warp per CTA-tier slot with the slot's global
// visited bitmap and queue.
// A step is a chain of two loads (the vertex's row, the picked in-neighbour);
// the next row is loaded while the visited check runs. The lane tiers keep
// their warps together: walks start and end in batches of kLtRefill lanes or
// more, and members are written out by the whole warp. Bound by that chain, at
// the slowest of 32 lanes' gathers about 1 us each. 2M samples of Chung-Lu 1M /
// 10M WC (18 members on average, 6 % of the walks above kLtQ): first tier 1.51
// -> .64 ms, second 1.13 -> .62; 500K of ER 10k / 100k (125 members) 1.2 (three
// passes) -> .29 and 24.5 -> 3.1. Batches of 4 or 12 lanes: within 2 %, of 1:
// .74 and .67; kLtQ 64 or 96 in blocks of 128: .96 and 1.10 for the first tier.
constexpr int kLtBlock = 256;
constexpr int kLtQ = 48;
constexpr int kLtRefill = 8;

__device__ __forceinline__ uint64_t lt_weight(uint32_t tau) { return tau == kSentinel ? (1ull << 32) : (uint64_t)tau; }

// step t of sample j from a vertex with in-row rw: the picked in-neighbour, or
// -1 when the walk ends there
__device__ __forceinline__ int32_t lt_step(const SampleArgs& a, uint64_t j, uint32_t t, const RowInfo& rw) {
    if (rw.deg == 0) return -1;
    const uint4 b = coin_block(a.rk, t, 0, kDomLt, j);
    const uint64_t U = (uint64_t)b.x | ((uint64_t)b.y << 32);
    const bool cond = t == 0 && !a.ris;
    uint32_t i;
    if (!a.lt_cum) {  // one weight w = tau a row, S = deg w
        if (cond) {
            i = (uint32_t)__umul64hi(U, rw.deg);  // floor(floor(U deg w / 2^64) / w)
        } else if (rw.tau == kSentinel) {  // w = 2^32
            i = 0;
        } else {
            if (b.x >= (uint64_t)rw.deg * rw.tau) return -1;  // no in-edge kept
            i = b.x / rw.tau;
        }
    } else {  // the first position whose running sum exceeds y
        const uint64_t base = a.lt_cum[rw.off];
        const uint64_t S = a.lt_cum[rw.off + rw.deg] - base;
        const uint64_t y = cond ? __umul64hi(U, S) : (uint64_t)b.x;  // cond: Pr[u] = w(u, v) / gamma_v
        if (!cond && y >= S) return -1;  // no in-edge kept
        uint32_t lo = 0, hi = rw.deg - 1;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (a.lt_cum[rw.off + mid + 1] - base > y) hi = mid;
            else lo = mid + 1;
        }
        i = lo;
    }
    return a.src[rw.off + i];
}

__device__ __forceinline__ uint32_t warp_incl_sum(uint32_t x) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, d);
        if ((threadIdx.x & 31) >= d) x += y;
    }
    return x;
}

// the lane whose run holds place idx of runs laid end to end (incl: this
// lane's inclusive end); all lanes call it
__device__ __forceinline__ int warp_owner(uint32_t incl, uint32_t idx) {
    int owner = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1)
        if (__shfl_sync(kFull, incl, owner + step - 1) <= idx) owner += step;
    return owner;
}

__device__ __forceinline__ void lt_header(const SampleArgs& a, uint64_t j, uint64_t at, uint32_t len, uint32_t v,
                                          uint64_t coins) {
    a.h_off[j - a.id_base] = at;
    a.h_len[j - a.id_base] = len;
    a.h_src[j - a.id_base] = v;
    a.h_retries[j - a.id_base] = 0;
    a.h_coins[j - a.id_base] = coins;
}

// The members of a lane's walk stand four to a 16-byte word, the words of a
// lane one column further right each, so that a lane compares four members a
// load and the warp reads one walk's members, both without bank conflicts. A
// new member whose hashed bit (of 128) is clear needs no search.
__global__ void __launch_bounds__(kLtBlock, 4) k_lt_walk(SampleArgs a) {
    __shared__ int4 s_q[kLtBlock / 32][kLtQ / 4][32];
    const int lane = threadIdx.x & 31;
    int4* const words = s_q[threadIdx.x >> 5][0];
    int32_t* const flat = reinterpret_cast<int32_t*>(words);
    auto word = [](int l, uint32_t c) { return c * 32 + (((uint32_t)l + c) & 31u); };
    const uint64_t count = input_count(a);
    bool busy = false, done = false, exhausted = false;
    uint64_t j = 0, coins = 0, sig0 = 0, sig1 = 0;
    uint32_t v = 0, len = 0, t = 0;
    RowInfo row = {};
    // up to 32 sources drawn together, one a lane
    uint64_t pool_base = 0;
    uint32_t pool_n = 0, pool_used = 0, p_v = 0;
    RowInfo p_row = {};
    uint64_t chunk_pos = 0, chunk_end = 0;
    uint32_t chunk = kLaneArenaChunk;

    auto add = [&](int32_t u) {  // member len of this lane's walk
        const uint32_t h = ((uint32_t)u * 0x9E3779B9u) >> 25;
        const uint64_t bit = 1ull << (h & 63u);
        if (h < 64u) sig0 |= bit;
        else sig1 |= bit;
        const uint32_t w = word(lane, len >> 2);
        if ((len & 3u) == 0) words[w] = make_int4(u, -1, -1, -1);
        else flat[4 * w + (len & 3u)] = u;
        ++len;
    };

    for (;;) {
        const unsigned dn = __ballot_sync(kFull, done);
        const unsigned free_l = __ballot_sync(kFull, !busy || done);
        if (__popc(free_l) >= kLtRefill || free_l == kFull) {
            if (dn) {
                const uint32_t mylen = done ? len : 0u;
                const uint32_t incl = warp_incl_sum(mylen);
                const uint32_t total = __shfl_sync(kFull, incl, 31);
                bool fits = true;
                if (chunk_end - chunk_pos < total) {
                    const uint64_t size = max((uint64_t)chunk, (uint64_t)total);
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(a.arena_cursor, (unsigned long long)size);
                    base = __shfl_sync(kFull, base, 0);
                    if (base + size > a.arena_cap) {
                        fits = false;
                        chunk = 0;
                        chunk_pos = chunk_end = 0;
                    } else {
                        chunk_pos = base;
                        chunk_end = base + size;
                    }
                }
                if (done) {
                    if (fits) lt_header(a, j, chunk_pos + (incl - mylen), len, v, coins);
                    else arena_overflow(a, j);
                    busy = done = false;
                }
                __syncwarp();
                if (fits) {
                    for (uint32_t b0 = 0; b0 < total; b0 += 32) {
                        const uint32_t idx = b0 + (uint32_t)lane;
                        const int owner = warp_owner(incl, idx);
                        const uint32_t i = idx - __shfl_sync(kFull, incl - mylen, owner);
                        if (idx < total) {
                            const int32_t u = flat[4 * word(owner, i >> 2) + (i & 3u)];
                            a.arena[chunk_pos + idx] = u;
                            count_member(a, u);
                        }
                    }
                    chunk_pos += total;
                }
                __syncwarp();
            }
            unsigned idle = __ballot_sync(kFull, !busy);
            while (idle && !exhausted) {
                if (pool_used == pool_n) {
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(a.work, 32ull);
                    base = __shfl_sync(kFull, base, 0);
                    if (base >= count) {
                        exhausted = true;
                        break;
                    }
                    pool_base = base;
                    pool_n = (uint32_t)min((unsigned long long)32, count - base);
                    pool_used = 0;
                    if ((uint32_t)lane < pool_n) {
                        p_v = draw_source<true>(a, input_id(a, base + lane));
                        p_row = a.rows[p_v];
                    }
                }
                const uint32_t take = min((uint32_t)__popc(idle), pool_n - pool_used);
                const uint32_t rank = __popc(idle & lanemask_lt());
                const int from = (int)min(pool_used + rank, 31u);
                const uint32_t n_v = __shfl_sync(kFull, p_v, from);
                RowInfo n_row;
                n_row.off = shfl_u64(p_row.off, from);
                n_row.deg = __shfl_sync(kFull, p_row.deg, from);
                n_row.tau = __shfl_sync(kFull, p_row.tau, from);
                if (!busy && rank < take) {
                    j = input_id(a, pool_base + pool_used + rank);
                    v = n_v;
                    row = n_row;
                    len = t = 0;
                    coins = sig0 = sig1 = 0;
                    busy = true;
                    add((int32_t)v);
                }
                pool_used += take;
                idle = __ballot_sync(kFull, !busy);
            }
            if (!__any_sync(kFull, busy)) {
                if (exhausted) break;
                continue;
            }
        }
        if (!busy || done) continue;  // the lane waits for the next batch
        coins += row.deg;
        const int32_t u = lt_step(a, j, t, row);
        ++t;
        if (u < 0) {
            done = true;
            continue;
        }
        row = a.rows[u];  // in flight during the visited check
        const uint32_t h = ((uint32_t)u * 0x9E3779B9u) >> 25;
        bool seen = false;
        if (((h < 64u ? sig0 : sig1) >> (h & 63u)) & 1ull) {
            for (uint32_t c = 0; c * 4 < len && !seen; ++c) {
                const int4 m = words[word(lane, c)];
                seen = m.x == u || m.y == u || m.z == u || m.w == u;
            }
        }
        if (seen) {
            done = true;  // the walk closes on R_j
        } else if (len == (uint32_t)kLtQ) {
            hand_on(a, j);  // a long walk: the next tier redraws it
            busy = false;
        } else {
            add(u);
        }
    }
}

// Medium LT walks: a lane a walk, its members listed in global memory and in
// an open-addressing visited table there, at most half full. Which slots are
// taken stands in a shared bitmap, which alone is cleared between walks, and a
// second bitmap by another hash tells most new vertices: a slot is read only
// where both bits are set (the tables of 77,824 lanes are 640 MB, so a read is
// a DRAM latency for the whole warp: .78 ms without the second bitmap, .62 with
// it, 1.13 with tables read at each probe and restored slot by slot). A walk
// longer than kLtMidCap is handed on.
constexpr int kLtMidBlock = 128;
constexpr int kLtMidBlocks = 4;  // an SM: 48 KB of bitmaps a block
constexpr uint32_t kLtMidHash = 2048;
constexpr uint32_t kLtMidBloom = 1024;
constexpr uint32_t kLtMidCap = 1024;

__global__ void __launch_bounds__(kLtMidBlock) k_lt_mid(SampleArgs a, uint32_t* __restrict__ hash_all,
                                                        int32_t* list_all) {
    __shared__ uint32_t s_occ[kLtMidBlock / 32][(kLtMidHash + kLtMidBloom) / 32][32];
    const int lane = threadIdx.x & 31;
    const uint64_t me = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t* const hash = hash_all + me * kLtMidHash;
    int32_t* const list = list_all + me * kLtMidCap;
    const int32_t* const warp_list = list_all + (me - lane) * kLtMidCap;
    uint32_t(*const occ)[32] = s_occ[threadIdx.x >> 5];  // word w of this lane's bitmap: occ[w][lane]
    uint32_t(*const bloom)[32] = occ + kLtMidHash / 32;
    auto bloom_bit = [](uint32_t u) { return (u * 0x9E3779B9u) >> 22; };
    static_assert(kLtMidBloom == 1u << 10, "bloom_bit: ten bits");
    const uint64_t count = input_count(a);
    bool busy = false, done = false, exhausted = false;
    uint64_t j = 0, coins = 0;
    uint32_t v = 0, len = 0, t = 0;
    RowInfo row = {};

    for (;;) {
        const unsigned dn = __ballot_sync(kFull, done);
        const unsigned free_l = __ballot_sync(kFull, !busy || done);
        if (__popc(free_l) >= kLtRefill || free_l == kFull) {
            if (dn) {
                const uint32_t mylen = done ? len : 0u;
                const uint32_t incl = warp_incl_sum(mylen);
                const uint32_t total = __shfl_sync(kFull, incl, 31);
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(a.arena_cursor, (unsigned long long)total);
                base = __shfl_sync(kFull, base, 0);
                const bool fits = base + total <= a.arena_cap;
                if (done) {
                    if (fits) lt_header(a, j, base + (incl - mylen), len, v, coins);
                    else arena_overflow(a, j);
                    busy = done = false;
                }
                __syncwarp();
                for (uint32_t b0 = 0; fits && b0 < total; b0 += 128) {
                    int32_t u[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {  // four loads in flight
                        const uint32_t idx = b0 + 32 * k + (uint32_t)lane;
                        const int owner = warp_owner(incl, idx);
                        const uint32_t i = idx - __shfl_sync(kFull, incl - mylen, owner);
                        u[k] = idx < total ? warp_list[owner * kLtMidCap + i] : 0;
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t idx = b0 + 32 * k + (uint32_t)lane;
                        if (idx < total) {
                            a.arena[base + idx] = u[k];
                            count_member(a, u[k]);
                        }
                    }
                }
                __syncwarp();
            }
            const unsigned idle = __ballot_sync(kFull, !busy);
            if (!exhausted) {
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(a.work, (unsigned long long)__popc(idle));
                base = __shfl_sync(kFull, base, 0);
                if (base + __popc(idle) >= count) exhausted = true;
                const uint64_t ti = base + __popc(idle & lanemask_lt());
                if (!busy && ti < count) {
                    j = input_id(a, ti);
                    v = draw_source(a, j);
                    row = a.rows[v];
#pragma unroll 8
                    for (uint32_t w = 0; w < (kLtMidHash + kLtMidBloom) / 32; ++w) occ[w][lane] = 0;
                    const uint32_t h = (v * 2654435761u) & (kLtMidHash - 1);
                    occ[h >> 5][lane] = 1u << (h & 31u);
                    const uint32_t b = bloom_bit(v);
                    bloom[b >> 5][lane] = 1u << (b & 31u);
                    hash[h] = v;
                    list[0] = (int32_t)v;
                    len = 1;
                    t = 0;
                    coins = 0;
                    busy = true;
                }
            }
            if (!__any_sync(kFull, busy)) {
                if (exhausted) break;
                continue;
            }
        }
        if (!busy || done) continue;  // the lane waits for the next batch
        coins += row.deg;
        const int32_t u = lt_step(a, j, t, row);
        ++t;
        if (u < 0) {
            done = true;
            continue;
        }
        row = a.rows[u];  // in flight during the visited check
        uint32_t g = ((uint32_t)u * 2654435761u) & (kLtMidHash - 1);
        const uint32_t b = bloom_bit((uint32_t)u);
        const bool maybe = (bloom[b >> 5][lane] >> (b & 31u)) & 1u;
        bool seen = false;
        while ((occ[g >> 5][lane] >> (g & 31u)) & 1u) {  // the table is at most half full: the probe ends
            if (maybe && hash[g] == (uint32_t)u) { seen = true; break; }
            g = (g + 1) & (kLtMidHash - 1);
        }
        if (seen) {
            done = true;
        } else if (len == kLtMidCap) {
            hand_on(a, j);
            busy = false;
        } else {
            occ[g >> 5][lane] |= 1u << (g & 31u);
            bloom[b >> 5][lane] |= 1u << (b & 31u);
            hash[g] = (uint32_t)u;
            list[len++] = u;
        }
    }
}

// Long LT walks: one warp per slot; lane 0 walks with the slot's global
// visited bitmap and queue, the warp copies the members out and clears the
// bitmap.
__global__ void __launch_bounds__(32) k_lt_long(SampleArgs a) {
    const int lane = threadIdx.x & 31;
    uint32_t* bitmap = a.bitmaps + (uint64_t)blockIdx.x * a.bitmap_words;
    int32_t* queue = a.queues + (uint64_t)blockIdx.x * a.queue_cap;
    const uint64_t count = input_count(a);
    for (;;) {
        unsigned long long ti = 0;
        if (lane == 0) ti = atomicAdd(a.work, 1ull);
        ti = __shfl_sync(kFull, ti, 0);
        if (ti >= count) break;
        const uint64_t j = input_id(a, ti);
        uint32_t len = 0, v = 0, outgrown = 0;
        uint64_t coins = 0;
        if (lane == 0) {
            v = draw_source(a, j);
            bitmap[v >> 5] |= 1u << (v & 31);
            queue[0] = (int32_t)v;
            len = 1;
            RowInfo rw = a.rows[v];
            for (uint32_t t = 0;; ++t) {  // at most n steps: each adds a new member
                coins += rw.deg;
                const int32_t u = lt_step(a, j, t, rw);
                if (u < 0) break;
                rw = a.rows[u];  // in flight during the visited check
                const uint32_t bit = 1u << (u & 31);
                if (bitmap[(uint32_t)u >> 5] & bit) break;
                if (len == a.queue_cap) {  // the walk outgrew the slot's queue
                    outgrown = 1;
                    break;
                }
                bitmap[(uint32_t)u >> 5] |= bit;
                queue[len++] = u;
            }
        }
        __syncwarp();
        len = __shfl_sync(kFull, len, 0);
        v = __shfl_sync(kFull, v, 0);
        coins = __shfl_sync(kFull, coins, 0);
        outgrown = __shfl_sync(kFull, outgrown, 0);
        unsigned long long base = 0;
        if (lane == 0 && !outgrown) base = atomicAdd(a.arena_cursor, (unsigned long long)len);
        base = __shfl_sync(kFull, base, 0);
        const bool fits = !outgrown && base + len <= a.arena_cap;
        for (uint32_t i = lane; i < len; i += 32) {
            const int32_t u = queue[i];
            if (fits) {
                a.arena[base + i] = u;
                count_member(a, u);
            }
            bitmap[(uint32_t)u >> 5] = 0;  // restore the all-zero bitmap
        }
        if (lane == 0) {
            if (fits) {
                a.h_off[j - a.id_base] = base;
                a.h_len[j - a.id_base] = len;
                a.h_src[j - a.id_base] = v;
                a.h_retries[j - a.id_base] = 0;
                a.h_coins[j - a.id_base] = coins;
            } else if (outgrown) {  // to the pass whose slots hold n-entry queues
                if (a.out_ids) hand_on(a, j);
                else atomicOr(&a.status->flags, kStListFull);
            } else {
                arena_overflow(a, j);
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ host
#define SK_CUDA(call)                                                                   \
    do {                                                                                \
        cudaError_t _e = (call);                                                        \
        if (_e != cudaSuccess) {                                                        \
            *err = std::string("CUDA error in skis_sample: ") + cudaGetErrorString(_e); \
            return _e == cudaErrorMemoryAllocation ? SKIS_ENOMEM : SKIS_ERR_CUDA;       \
        }                                                                               \
    } while (0)

template <typename T>
static cudaError_t grow_copy(T** p, uint64_t old_n, uint64_t new_n, cudaStream_t st) {
    T* q = nullptr;
    cudaError_t e = dev_alloc_t(&q, (size_t)new_n, st);
    if (e != cudaSuccess) return e;
    if (*p && old_n) {
        e = cudaMemcpyAsync(q, *p, old_n * sizeof(T), cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) { dev_free(q, st); return e; }
    }
    dev_free(*p, st);
    *p = q;
    return cudaSuccess;
}

// threads of the CTA-tier blocks that the slots are counted for (launch_cta)
static int cta_block(const skis_sketch* s) { return s->cta_threads ? s->cta_threads : kCtaBlock; }

// Arena entries a sketch's first `count` samples get: room for samples of 128
// members within 2 GiB, at least 8 a sample. Sizes run from 4 members a sample
// (trivalency) to 60-75 (weighted cascade, LT 18), and a pass that overflows
// draws what did not fit again.
static uint64_t first_arena(uint64_t count) {
    return std::max<uint64_t>({count * 8, std::min<uint64_t>(count * 128, 1u << 29), 1u << 20});
}

// Entries that `count` more samples are given: what the samples so far had, as
// far as it is known. The entries they reserved are no fewer than their members,
// and more by the unused ends of the warps' chunks, at most arena_ends; a first
// allotment's size is taken within these two. (By the reserved entries alone, a
// call for one sample, which opens a chunk for it, made the next call of 10M
// samples ask for 115 GB.)
static uint64_t more_arena(const skis_sketch* s, uint64_t count, uint64_t used) {
    const double c = 1.125 * (double)count / (double)std::max<uint64_t>(s->arena_drawn, 1);
    const double least = c * (double)(used - std::min(used, s->arena_ends)), most = c * (double)used;
    return (uint64_t)std::min(std::max(least, std::min(most, (double)first_arena(count))), (double)(1ull << 50));
}

// slack: arena entries that the tiers' warps may leave unused at the ends of their chunks;
// warps: the warp tier's warps (0: no such tier)
static int ensure_sample_buffers(skis_sketch* s, uint64_t count, uint64_t slack, uint64_t warps, cudaStream_t st,
                                 std::string* err) {
    const skis_graph* g = s->g;
    // each buffer is asked for by its own pointer (or a size that is reset before
    // its group is freed), so that after an allocation failed the next call finds
    // out which are missing
    if (!s->ctr) {
        SK_CUDA(dev_alloc_t(&s->ctr, 1, st));
        SK_CUDA(cudaMemsetAsync(s->ctr, 0, sizeof(SampleCounters), st));
    }
    if (!s->status) SK_CUDA(dev_alloc_t(&s->status, 1, st));
    for (int i = 0; i < 4; ++i)
        if (!s->ev[i]) SK_CUDA(cudaEventCreate(&s->ev[i]));
    const uint64_t need = s->T + count;
    if (need > s->hcap) {
        const uint64_t nc = std::max<uint64_t>(need, s->hcap * 2);
        SK_CUDA(grow_copy(&s->h_off, s->T, nc, st));
        SK_CUDA(grow_copy(&s->h_len, s->T, nc, st));
        SK_CUDA(grow_copy(&s->h_src, s->T, nc, st));
        SK_CUDA(grow_copy(&s->h_retries, s->T, nc, st));
        SK_CUDA(grow_copy(&s->h_coins, s->T, nc, st));
        s->hcap = nc;
    }
    if (count > s->list_cap) {
        s->list_cap = 0;
        dev_free(s->to_warp_ids, st);
        dev_free(s->to_cta_ids, st);
        dev_free(s->big_ids, st);
        dev_free(s->ovf_ids[0], st);
        dev_free(s->ovf_ids[1], st);
        s->to_warp_ids = s->to_cta_ids = s->big_ids = s->ovf_ids[0] = s->ovf_ids[1] = nullptr;
        SK_CUDA(dev_alloc_t(&s->to_warp_ids, (size_t)count, st));
        SK_CUDA(dev_alloc_t(&s->to_cta_ids, (size_t)count, st));
        SK_CUDA(dev_alloc_t(&s->big_ids, (size_t)count, st));
        SK_CUDA(dev_alloc_t(&s->ovf_ids[0], (size_t)count, st));
        SK_CUDA(dev_alloc_t(&s->ovf_ids[1], (size_t)count, st));
        dev_free(s->srcrec, st);
        dev_free(s->srcpick, st);
        s->srcrec = nullptr;
        s->srcpick = nullptr;
        SK_CUDA(dev_alloc_t(&s->srcrec, (size_t)count, st));
        SK_CUDA(dev_alloc_t(&s->srcpick, (size_t)count, st));
        s->list_cap = count;
    }
    if (!s->arena) {
        uint64_t cap = s->arena_hint;
        if (!cap) cap = s->lean ? std::max<uint64_t>(count * 8, 1u << 20) : first_arena(count) + slack;
        SK_CUDA(dev_alloc_t(&s->arena, (size_t)cap, st));
        s->arena_cap = cap;
    } else if (s->T > 0) {
        // more samples like the ones so far: the arena grows before the pass
        // when they would not fit (or, without the memory now, as it overflows)
        const uint64_t used = std::min(s->arena_used, s->arena_cap);
        const uint64_t want = used + more_arena(s, count, used) + slack;
        if (want > s->arena_cap) {
            const cudaError_t e = grow_copy(&s->arena, used, std::max(want, s->arena_cap * 2), st);
            if (e == cudaSuccess) s->arena_cap = std::max(want, s->arena_cap * 2);
            else if (e != cudaErrorMemoryAllocation) SK_CUDA(e);
        }
    }
    if (g->lt) {  // medium LT walks: one table and list per lane
        s->lt_mid_lanes = (uint64_t)std::max(1, (sm_count() * kLtMidBlocks) >> s->lean) * kLtMidBlock;
        if (!s->lt_hash) SK_CUDA(dev_alloc_t(&s->lt_hash, (size_t)(s->lt_mid_lanes * kLtMidHash), st));
        if (!s->lt_list) SK_CUDA(dev_alloc_t(&s->lt_list, (size_t)(s->lt_mid_lanes * kLtMidCap), st));
    }
    if (warps > s->spill_warps) {  // warp tier: a spill slot a warp
        dev_free(s->spill_hash, st);
        dev_free(s->spill_queue, st);
        s->spill_hash = nullptr;
        s->spill_queue = nullptr;
        s->spill_warps = 0;
        SK_CUDA(dev_alloc_t(&s->spill_hash, (size_t)(warps << spill_size(g->n).hash_bits), st));
        SK_CUDA(dev_alloc_t(&s->spill_queue, (size_t)(warps * spill_size(g->n).cap), st));
        s->spill_warps = warps;
    }
    // CTA-tier slots: an n-bit visited bitmap and a queue of min(n, cta_queue_cap)
    // entries each (a sample with more members moves to a pass over slots with
    // n-entry queues), 1024 threads of blocks per SM within ~12 GB. A block
    // clears its bitmap when it takes its first sample (few of them do where few
    // samples come this far)
    const uint32_t qcap = (uint32_t)std::min<uint64_t>((uint64_t)g->n, s->cta_queue_cap);
    int slots = s->cta_slots;
    if (slots <= 0) {
        const uint64_t per_slot = (uint64_t)qcap * 4 + ((uint64_t)g->n + 31) / 32 * 4;
        const uint64_t budget = 12ull << 30;
        const uint64_t per_sm = g->lt ? 2 : 1024 / cta_block(s);
        slots = (int)std::min<uint64_t>((uint64_t)sm_count() * per_sm, std::max<uint64_t>(1, budget / per_slot));
        slots = std::max(1, slots >> s->lean);
    }
    if (slots != s->cta_slots_alloc || qcap != s->queue_cap) {
        dev_free(s->bitmaps, st);
        dev_free(s->queues, st);
        dev_free(s->slot_clean, st);
        dev_free(s->big_queues, st);  // the pass for outgrown samples uses the first slots' bitmaps: as many at most
        s->bitmaps = s->slot_clean = nullptr;
        s->queues = s->big_queues = nullptr;
        s->cta_slots_alloc = s->big_slots = 0;
        s->bitmap_words = ((uint64_t)g->n + 31) / 32;
        SK_CUDA(dev_alloc_t(&s->bitmaps, (size_t)(s->bitmap_words * slots), st));
        SK_CUDA(dev_alloc_t(&s->slot_clean, (size_t)slots, st));
        if (g->lt) SK_CUDA(cudaMemsetAsync(s->bitmaps, 0, s->bitmap_words * slots * sizeof(uint32_t), st));
        else SK_CUDA(cudaMemsetAsync(s->slot_clean, 0, (size_t)slots * sizeof(uint32_t), st));
        SK_CUDA(dev_alloc_t(&s->queues, (size_t)((uint64_t)qcap * slots), st));
        s->cta_slots_alloc = slots;
        s->queue_cap = qcap;
    }
    return SKIS_OK;
}

// The pass over samples that outgrew a CTA-tier slot's queue: slots with
// n-entry queues (their bitmaps are the first slots' of the CTA tier, all
// zero between launches), allocated on first use within ~8 GB.
static int ensure_big_slots(skis_sketch* s, cudaStream_t st, std::string* err) {
    if (s->big_queues) return SKIS_OK;
    const uint64_t n = (uint64_t)s->g->n;
    const uint64_t budget = 8ull << 30;
    int slots = (int)std::min<uint64_t>((uint64_t)s->cta_slots_alloc, std::max<uint64_t>(1, budget / (n * 4)));
    slots = std::max(1, slots >> s->lean);
    SK_CUDA(dev_alloc_t(&s->big_queues, (size_t)(n * slots), st));
    s->big_slots = slots;
    return SKIS_OK;
}

// At most `slots` blocks of kCtaThreads, for a count in (above, upto] or for any other.
template <int kCtaThreads>
static void launch_cta_blocks(const SampleArgs& a, int slots, uint64_t above, uint64_t upto, bool within,
                              cudaStream_t st) {
    k_iis_cta<kCtaThreads><<<std::min(slots, sm_count() * (1024 / kCtaThreads)), kCtaThreads, 0, st>>>(a, above, upto,
                                                                                                      within);
    note_launch();
}

// The CTA tier for a pass of `pass` samples; how many of them come here is on
// the device, so a pass that two block sizes may take is launched with both,
// one of which ends at once.
static void launch_cta(const skis_sketch* s, const SampleArgs& a, int slots, uint64_t pass, cudaStream_t st) {
    const uint64_t share = pass / kCtaHubShare;
    const uint64_t few = kCtaFew * (uint64_t)sm_count(), many = kCtaMany * (uint64_t)sm_count();
    if (s->cta_threads == 512) {
        k_iis_cta<512><<<slots, 512, 0, st>>>(a, 0, ~0ull, true);
        note_launch();
    } else if (s->cta_threads == 256) {
        k_iis_cta<256><<<slots, 256, 0, st>>>(a, 0, ~0ull, true);
        note_launch();
    } else if (share >= many) {
        launch_cta_blocks<kCtaBlock>(a, slots, 0, ~0ull, true, st);
    } else {
        if (pass <= few) launch_cta_blocks<512>(a, slots, share, many, true, st);
        else launch_cta_blocks<256>(a, slots, share, many, true, st);
        launch_cta_blocks<kCtaBlock>(a, slots, share, many, false, st);
    }
}

static int occupancy_grid(const void* kernel, int threads, int override_blocks, uint64_t max_useful,
                          std::string* err, int* out) {
    int blocks = override_blocks;
    if (blocks <= 0) {
        int per_sm = 0;
        SK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0));
        blocks = sm_count() * std::max(per_sm, 1);
    }
    *out = (int)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)blocks, max_useful));
    return SKIS_OK;
}

static int sample_passes(skis_sketch* s, uint64_t count, cudaStream_t st, std::string* err) {
    const skis_graph* g = s->g;
    if (g->W == 0 && !s->ris) {
        *err = "skis_sample: Gamma = 0, the graph has no non-singular sample";
        return SKIS_EINVAL;
    }
    if (count == 0) return SKIS_OK;
    const bool thread_tier = s->thread_max_deg > 0;
    int warp_blocks = 0, lane_blocks = 0, lt_blocks = 0;
    int rc = occupancy_grid((const void*)k_iis_lane, kLaneBlock, s->thread_blocks,
                        (count + kLaneBlock - 1) / kLaneBlock, err, &lane_blocks);
    if (rc != SKIS_OK) return rc;
    // no more blocks than can be resident (every warp holds a spill slot) and
    // no more warps than samples
    rc = occupancy_grid((const void*)k_iis_warp, kWarpThreads, 0,
                        (count + kWarpThreads / 32 - 1) / (kWarpThreads / 32), err, &warp_blocks);
    if (rc != SKIS_OK) return rc;
    if (s->warp_blocks > 0) warp_blocks = std::min(warp_blocks, s->warp_blocks);
    warp_blocks = std::max(1, warp_blocks >> s->lean);
    if (g->lt) {
        rc = occupancy_grid((const void*)k_lt_walk, kLtBlock, s->thread_blocks, (count + kLtBlock - 1) / kLtBlock,
                            err, &lt_blocks);
        if (rc != SKIS_OK) return rc;
    }
    // every warp's open chunk (a warp without a sample opens none)
    const uint64_t lane_warps = (uint64_t)(g->lt ? lt_blocks : lane_blocks) * (kLaneBlock / 32);
    const uint64_t warps = g->lt ? 0 : (uint64_t)warp_blocks * (kWarpThreads / 32);
    static_assert(kLaneBlock == kLtBlock, "one block size for both lane tiers");
    const uint64_t slack = kLaneArenaChunk * std::min(count, lane_warps) + kArenaChunk * std::min(count, warps);
    rc = ensure_sample_buffers(s, count, slack, warps, st, err);
    if (rc != SKIS_OK) return rc;

    SampleArgs base;
    base.alias = g->alias;
    base.rows = g->rows;
    base.src = g->src;
    base.tau = g->row_uniform ? nullptr : g->tau;
    base.n = (uint64_t)g->n;
    base.W = g->W;
    base.seed = s->seed;
    base.rk = philox_keys(s->seed);
    base.retry_cap = s->retry_cap;
    base.max_deg = s->thread_max_deg;
    base.max_steps = s->thread_max_steps;
    base.max_retries = s->thread_max_retries;
    base.warp_max_coins = s->warp_max_coins;
    base.cta_hub_quads = s->cta_hub_quads;
    base.ris = s->ris;
    base.ids = nullptr;
    base.first_id = s->id_base + s->T;
    base.id_base = s->id_base;
    base.count = count;
    base.count_dev = nullptr;
    base.arena_cursor = &s->ctr->arena;
    base.novf = &s->ctr->novf;
    base.h_off = s->h_off;
    base.h_len = s->h_len;
    base.h_src = s->h_src;
    base.h_retries = s->h_retries;
    base.h_coins = s->h_coins;
    base.arena = s->arena;
    base.arena_cap = s->arena_cap;
    base.status = s->status;
    base.bitmaps = s->bitmaps;
    base.slot_clean = s->slot_clean;
    base.queues = s->queues;
    base.bitmap_words = s->bitmap_words;
    base.queue_cap = s->queue_cap;
    base.srcrec = nullptr;
    base.srcpick = nullptr;
    base.up_rec = nullptr;
    base.up_pick = nullptr;
    base.up_first = 0;
    base.up_count = 0;
    base.lt_cum = g->lt_cum;
    base.spill_hash = s->spill_hash;
    base.spill_queue = s->spill_queue;
    base.spill = spill_size(g->n);
    // per-vertex member counts, kept while they describe exactly samples
    // [0, T): invalid until this call succeeds
    const bool counting = s->vcount_ok && s->vcount_T == s->T;
    base.vcount = nullptr;
    if (counting) {
        if (!s->vcount) {
            SK_CUDA(dev_alloc_t(&s->vcount, (size_t)g->n, st));
            SK_CUDA(cudaMemsetAsync(s->vcount, 0, (size_t)g->n * sizeof(uint32_t), st));
        }
        base.vcount = s->vcount;
    }
    s->vcount_ok = false;
    base.chain = nullptr;
    if (s->bucket && !s->ris && !g->lt) {
        rc = graph_ensure_chain(g, st, err);
        if (rc != SKIS_OK) return rc;
        base.chain = g->chain;
    }
    DevStatus hst;
    SampleCounters hc;
    int pass = 0;
    s->last_thread_ms = s->last_warp_ms = s->last_cta_ms = s->last_sample_ms = 0;
    s->last_to_warp = s->last_deferred = 0;
    s->last_passes = 0;
    SK_CUDA(cudaMemsetAsync(s->status, 0, sizeof(DevStatus), st));
    SK_CUDA(cudaMemsetAsync(&s->status->first_bad, 0xFF, sizeof(unsigned long long), st));
    for (;;) {
        base.ovf_ids = s->ovf_ids[pass & 1];
        // reset every per-pass cursor and count; the arena cursor persists
        SK_CUDA(cudaMemsetAsync(&s->ctr->novf, 0, sizeof(SampleCounters) - sizeof(unsigned long long), st));
        SampleArgs at = base, aw = base, ac = base;
        // thread tier: the input ids; hands on to the warp tier
        at.work = &s->ctr->work_thread;
        at.out_ids = s->to_warp_ids;
        at.out_count = &s->ctr->n_to_warp;
        // warp tier: the thread tier's hand-ons (or the input ids without it)
        if (thread_tier) {
            aw.ids = s->to_warp_ids;
            aw.count_dev = &s->ctr->n_to_warp;
        }
        aw.work = &s->ctr->work_warp;
        aw.out_ids = s->to_cta_ids;
        aw.out_count = &s->ctr->n_to_cta;
        // CTA tier: the warp tier's hand-ons
        ac.ids = s->to_cta_ids;
        ac.count_dev = &s->ctr->n_to_cta;
        ac.work = &s->ctr->work_cta;
        ac.out_ids = s->big_ids;  // samples that outgrow a slot's queue
        ac.out_count = &s->ctr->n_big;

        SK_CUDA(cudaEventRecord(s->ev[0], st));
        if (g->lt) {  // LT: lane-per-sample walks, lane-per-walk medium walks, long walks on the slots
            aw.ids = s->to_warp_ids;
            aw.count_dev = &s->ctr->n_to_warp;
            k_lt_walk<<<lt_blocks, kLtBlock, 0, st>>>(at); note_launch();
            SK_CUDA(cudaGetLastError());
            SK_CUDA(cudaEventRecord(s->ev[1], st));
            k_lt_mid<<<s->lt_mid_lanes / kLtMidBlock, kLtMidBlock, 0, st>>>(aw, s->lt_hash, s->lt_list);
            note_launch();
            SK_CUDA(cudaGetLastError());
            SK_CUDA(cudaEventRecord(s->ev[2], st));
            k_lt_long<<<s->cta_slots_alloc, 32, 0, st>>>(ac); note_launch();
            SK_CUDA(cudaGetLastError());
            SK_CUDA(cudaEventRecord(s->ev[3], st));
        } else {
            if (thread_tier) {
                const uint64_t in_count = base.count;
                k_sources<<<(int)std::max<uint64_t>(1, std::min<uint64_t>((in_count + 255) / 256, (uint64_t)sm_count() * 16)),
                            256, 0, st>>>(at, s->srcrec, s->srcpick); note_launch();
                at.srcrec = s->srcrec;
                at.srcpick = base.chain ? s->srcpick : nullptr;
                if (!base.ids) {  // contiguous ids: later tiers find their samples' records by id
                    aw.up_rec = ac.up_rec = s->srcrec;
                    aw.up_pick = ac.up_pick = at.srcpick;
                    aw.up_first = ac.up_first = base.first_id;
                    aw.up_count = ac.up_count = base.count;
                }
                k_iis_lane<<<lane_blocks, kLaneBlock, 0, st>>>(at); note_launch();
                SK_CUDA(cudaGetLastError());
            }
            SK_CUDA(cudaEventRecord(s->ev[1], st));
            k_iis_warp<<<warp_blocks, kWarpThreads, 0, st>>>(aw); note_launch();
            SK_CUDA(cudaGetLastError());
            SK_CUDA(cudaEventRecord(s->ev[2], st));
            launch_cta(s, ac, s->cta_slots_alloc, base.count, st);
            SK_CUDA(cudaGetLastError());
            SK_CUDA(cudaEventRecord(s->ev[3], st));
        }
        SK_CUDA(cudaMemcpyAsync(&hc, s->ctr, sizeof(SampleCounters), cudaMemcpyDeviceToHost, st));
        SK_CUDA(cudaMemcpyAsync(&hst, s->status, sizeof(DevStatus), cudaMemcpyDeviceToHost, st));
        SK_CUDA(cudaStreamSynchronize(st));
        float ms_t = 0, ms_w = 0, ms_c = 0, ms_b = 0;
        cudaEventElapsedTime(&ms_t, s->ev[0], s->ev[1]);
        cudaEventElapsedTime(&ms_w, s->ev[1], s->ev[2]);
        cudaEventElapsedTime(&ms_c, s->ev[2], s->ev[3]);
        if (hc.n_big > 0) {  // samples that outgrew a slot's queue, on slots with n-entry queues
            rc = ensure_big_slots(s, st, err);
            if (rc != SKIS_OK) return rc;
            SampleArgs ab = ac;
            ab.ids = s->big_ids;
            ab.count_dev = &s->ctr->n_big;
            ab.work = &s->ctr->work_big;
            ab.queues = s->big_queues;
            ab.queue_cap = (uint32_t)g->n;
            ab.out_ids = nullptr;
            ab.out_count = nullptr;
            SK_CUDA(cudaEventRecord(s->ev[2], st));
            if (g->lt) {
                k_lt_long<<<s->big_slots, 32, 0, st>>>(ab); note_launch();
            } else {
                launch_cta(s, ab, s->big_slots, hc.n_big, st);
            }
            SK_CUDA(cudaGetLastError());
            SK_CUDA(cudaEventRecord(s->ev[3], st));
            SK_CUDA(cudaMemcpyAsync(&hc, s->ctr, sizeof(SampleCounters), cudaMemcpyDeviceToHost, st));
            SK_CUDA(cudaMemcpyAsync(&hst, s->status, sizeof(DevStatus), cudaMemcpyDeviceToHost, st));
            SK_CUDA(cudaStreamSynchronize(st));
            cudaEventElapsedTime(&ms_b, s->ev[2], s->ev[3]);
            ms_c += ms_b;
        }
        s->last_thread_ms += ms_t;
        s->last_warp_ms += ms_w;
        s->last_cta_ms += ms_c;
        s->last_sample_ms += ms_t + ms_w + ms_c;
        s->last_to_warp += (thread_tier || g->lt) ? hc.n_to_warp : count;
        s->last_deferred += hc.n_to_cta;
        s->last_passes += 1;
        if (hc.novf == 0) break;
        // some reservations did not fit: grow the arena (keeping every
        // completed sample, all of which lie below the old capacity) and
        // rerun exactly the samples that failed. The cursor counted every
        // reservation, placed or not, so what the rerun needs is known up to
        // the ends of chunks that a next sample does not fit in
        const uint64_t old_cap = s->arena_cap;
        uint64_t new_cap = std::max<uint64_t>(old_cap * 2, hc.arena + hc.arena / 8) + slack;
        cudaError_t e = grow_copy(&s->arena, old_cap, new_cap, st);
        if (e == cudaErrorMemoryAllocation)  // no room for all of it: what fits at twice the size, then further
            e = grow_copy(&s->arena, old_cap, new_cap = old_cap * 2, st);
        if (e != cudaSuccess) {
            *err = "skis_sample: the member arena could not grow to " + std::to_string(new_cap) + " entries";
            return SKIS_ERR_ARENA_FULL;
        }
        s->arena_cap = new_cap;
        unsigned long long cur = old_cap;
        SK_CUDA(cudaMemcpyAsync(&s->ctr->arena, &cur, sizeof(cur), cudaMemcpyHostToDevice, st));
        base.arena = s->arena;
        base.arena_cap = s->arena_cap;
        base.ids = s->ovf_ids[pass & 1];
        base.first_id = 0;
        base.count = hc.novf;
        ++pass;
    }
    s->T += count;
    s->arena_used = hc.arena;
    s->arena_drawn += count;
    s->arena_ends += slack * s->last_passes;
    if (counting) {
        s->vcount_ok = true;
        s->vcount_T = s->T;
    }
    if (hst.flags & kStListFull) {
        *err = "skis_sample: internal error: a sample outgrew a queue of n entries";
        return SKIS_ERR_INTERNAL;
    }
    if (hst.flags & kStRetry) {
        *err = "skis_sample: a conditioned first step reached the retry cap (" + std::to_string(s->retry_cap) +
               " rounds) at sample id " + std::to_string(hst.first_bad) + "; failed samples are empty";
        return SKIS_ERR_RETRY_LIMIT;
    }
    return SKIS_OK;
}

// The tiers' scratch, and an arena of the library's own choice that holds no
// sample yet.
bool sketch_release_scratch(skis_sketch* s, cudaStream_t st) {
    const bool any = s->spill_hash || s->bitmaps || s->queues || s->lt_hash || s->lt_list;
    dev_free(s->spill_hash, st);
    dev_free(s->spill_queue, st);
    dev_free(s->bitmaps, st);
    dev_free(s->slot_clean, st);
    dev_free(s->queues, st);
    dev_free(s->big_queues, st);
    dev_free(s->lt_hash, st);
    dev_free(s->lt_list, st);
    s->spill_hash = s->bitmaps = s->slot_clean = s->lt_hash = nullptr;
    s->spill_queue = s->queues = s->big_queues = s->lt_list = nullptr;
    s->spill_warps = 0;
    s->cta_slots_alloc = s->big_slots = 0;
    if (s->T == 0 && !s->arena_hint) {
        dev_free(s->arena, st);
        s->arena = nullptr;
        s->arena_cap = s->arena_used = 0;
    }
    dev_trim(st);
    return any;
}

// The passes of one call; where the device has no room for their scratch, again
// with half of the slots, spill slots and LT lanes each time, and room for 8
// members a sample at first (the sketch keeps to what was found). At half, all
// of it takes less than 608 CTA-tier slots within 8 GB did with blocks of 256.
int sketch_sample(skis_sketch* s, uint64_t count, cudaStream_t st, std::string* err) {
    constexpr int kLeanMost = 11;  // one slot, one block of warps
    const uint64_t T0 = s->T;
    const int lean0 = s->lean;
    for (;;) {
        const int rc = sample_passes(s, count, st, err);
        if (rc == SKIS_OK || s->T != T0) return rc;
        const bool again = (rc == SKIS_ENOMEM && s->lean < kLeanMost) || (rc == SKIS_ERR_ARENA_FULL && s->lean == lean0);
        if (again || s->lean != lean0) sketch_release_scratch(s, st);  // its sizes go by lean
        // a call that appended nothing: what its passes reserved is free again (and is
        // not taken for demand when a later call's overflow sizes the arena)
        if (s->T == 0) s->arena_used = 0;
        if (s->ctr)
            cudaMemcpyAsync(&s->ctr->arena, &s->arena_used, sizeof(s->arena_used), cudaMemcpyHostToDevice, st);
        if (!again) {
            s->lean = lean0;
            return rc;
        }
        ++s->lean;
        err->clear();
    }
}

// The one batch sample whose inclusive prefix of sizes first reaches need:
// pre is the exclusive scan with the total appended, so the index i with
// pre[i] < need <= pre[i + 1] is unique when pre[count] >= need.
__global__ void k_first_reach(const uint64_t* __restrict__ pre, uint64_t count, uint64_t need,
                              unsigned long long* __restrict__ out) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x)
        if (pre[i] < need && pre[i + 1] >= need) *out = i;
}

int sketch_sample_to_size(skis_sketch* s, uint64_t target, uint64_t max_count, cudaStream_t st, uint64_t* appended,
                          std::string* err) {
    *appended = 0;
    uint64_t cur = 0;  // sum of |R_j| over the samples already in the sketch
    if (s->T > 0) {
        uint64_t* pre = nullptr;
        SK_CUDA(dev_alloc_t(&pre, (size_t)s->T + 1, st));
        SK_CUDA(scan_u32_to_u64(s->h_len, pre, (int64_t)s->T, st));
        SK_CUDA(cudaMemcpyAsync(&cur, pre + s->T, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
        SK_CUDA(cudaStreamSynchronize(st));
        dev_free(pre, st);
    }
    while (cur < target && *appended < max_count) {
        const uint64_t need = target - cur;
        // batch: the expected count to reach the target at the sizes seen
        // so far, plus 5 %, within [2^16, what is left of max_count]
        uint64_t batch = 1u << 16;
        if (s->T > 0 && cur > 0) {
            const double mean = (double)cur / (double)s->T;
            batch = std::max<uint64_t>(batch, (uint64_t)((double)need / mean * 1.05) + 1024);
        }
        batch = std::min<uint64_t>(batch, max_count - *appended);
        const uint64_t T0 = s->T;
        int rc = sketch_sample(s, batch, st, err);
        if (rc != SKIS_OK) return rc;
        uint64_t* pre = nullptr;
        unsigned long long* d_at = nullptr;
        SK_CUDA(dev_alloc_t(&pre, (size_t)batch + 1, st));
        SK_CUDA(dev_alloc_t(&d_at, 1, st));
        SK_CUDA(scan_u32_to_u64(s->h_len + T0, pre, (int64_t)batch, st));
        SK_CUDA(cudaMemsetAsync(d_at, 0xFF, sizeof(unsigned long long), st));
        k_first_reach<<<(int)std::max<uint64_t>(1, std::min<uint64_t>((batch + 255) / 256, (uint64_t)sm_count() * 8)), 256, 0,
                        st>>>(pre, batch, need, d_at); note_launch();
        SK_CUDA(cudaGetLastError());
        uint64_t tot = 0;
        unsigned long long at = 0;
        SK_CUDA(cudaMemcpyAsync(&tot, pre + batch, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
        SK_CUDA(cudaMemcpyAsync(&at, d_at, sizeof(at), cudaMemcpyDeviceToHost, st));
        SK_CUDA(cudaStreamSynchronize(st));
        if (tot >= need) {
            uint64_t upto = 0;  // sizes of batch samples 0 .. at
            SK_CUDA(cudaMemcpyAsync(&upto, pre + at + 1, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
            SK_CUDA(cudaStreamSynchronize(st));
            s->T = T0 + at + 1;  // later samples of the batch are dropped
            s->vcount_ok = false;  // the counts include them
            *appended += at + 1;
            cur += upto;
        } else {
            *appended += batch;
            cur += tot;
        }
        dev_free(pre, st);
        dev_free(d_at, st);
    }
    return SKIS_OK;
}

// Autotuner of the tier split: pilot sampling of ids [0, pilot) on a scratch
// sketch under each candidate (thread-tier degree limit, step budget), best of
// two runs each, fastest kept. Samples do not depend on the split, so only
// time is compared.
int sketch_autotune(skis_sketch* s, uint64_t pilot, cudaStream_t st, double* cand_ms, int cand_cap, int* ncand,
                    std::string* err) {
    static const uint32_t kDeg[] = {0, 64, 128, 192, 256, 512};
    static const uint32_t kSteps[] = {128, 256, 1024};
    static const uint32_t kCoins[] = {4096, 16384, 65536, 262144};
    skis_sketch tmp;
    tmp.g = s->g;
    tmp.seed = s->seed;
    tmp.retry_cap = s->retry_cap;
    tmp.ris = s->ris;
    tmp.vcount_ok = false;
    tmp.bucket = s->bucket;
    tmp.thread_max_retries = s->thread_max_retries;
    tmp.warp_max_coins = s->warp_max_coins;
    tmp.cta_hub_quads = s->cta_hub_quads;
    tmp.cta_queue_cap = s->cta_queue_cap;
    tmp.cta_threads = s->cta_threads;
    tmp.cta_slots = s->cta_slots;
    tmp.warp_blocks = s->warp_blocks;
    tmp.thread_blocks = s->thread_blocks;
    tmp.stream = st;
    double best = 1e300;
    uint32_t best_deg = s->thread_max_deg, best_steps = s->thread_max_steps, best_coins = s->warp_max_coins;
    int k = 0, rc = SKIS_OK;
    // the pilot time of the current candidate (best of two runs)
    auto time_pilot = [&]() -> double {
        double ms = 1e300;
        for (int rep = 0; rep < 2 && rc == SKIS_OK; ++rep) {
            tmp.T = 0;
            if (tmp.ctr) {
                const cudaError_t e = cudaMemsetAsync(&tmp.ctr->arena, 0, sizeof(unsigned long long), st);
                if (e != cudaSuccess) { *err = cudaGetErrorString(e); rc = SKIS_ERR_CUDA; }
            }
            if (rc == SKIS_OK) rc = sketch_sample(&tmp, pilot, st, err);
            if (rc == SKIS_OK) ms = std::min(ms, tmp.last_sample_ms);
        }
        if (rc == SKIS_OK && cand_ms && k < cand_cap) cand_ms[k] = ms;
        ++k;
        return ms;
    };
    // first the lane/warp split, then the warp/CTA split under the chosen one
    for (uint32_t d : kDeg) {
        for (uint32_t m : kSteps) {
            if (d == 0 && m != kSteps[0]) continue;  // no thread tier: the budget is moot
            tmp.thread_max_deg = d;
            tmp.thread_max_steps = m;
            const double ms = time_pilot();
            if (rc != SKIS_OK) break;
            if (ms < best) {
                best = ms;
                best_deg = d;
                best_steps = m;
            }
        }
        if (rc != SKIS_OK) break;
    }
    tmp.thread_max_deg = best_deg;
    tmp.thread_max_steps = best_steps;
    for (uint32_t c : kCoins) {
        if (rc != SKIS_OK) break;
        tmp.warp_max_coins = c;
        const double ms = time_pilot();
        if (rc == SKIS_OK && ms < best) {
            best = ms;
            best_coins = c;
        }
    }
    sketch_release(&tmp);
    if (ncand) *ncand = k;
    if (rc != SKIS_OK) return rc;
    s->thread_max_deg = best_deg;
    s->thread_max_steps = best_steps;
    s->warp_max_coins = best_coins;
    return SKIS_OK;
}

}  // namespace skis
