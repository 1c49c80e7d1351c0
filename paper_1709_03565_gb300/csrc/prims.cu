// Device primitives used while building the graph and the greedy index:
// stream-ordered allocation, exclusive prefix sums (u32->u64, u64, u128),
// a stable LSD radix sort of the edges by (destination, source), and a u64
// sum.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "skis_internal.cuh"

namespace skis {

// --------------------------------------------------------------- launches
static std::atomic<uint64_t> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
uint64_t launches() { return g_launches.load(std::memory_order_relaxed); }

// ------------------------------------------------------------- allocation
static std::once_flag g_pool_once;
static std::atomic<uint64_t> g_allocs{0};
uint64_t allocations() { return g_allocs.load(std::memory_order_relaxed); }

// An allocation that failed is reported by its status alone: the runtime also
// keeps it as the thread's last error, where the next launch's check, on this
// call or a later one, would find it and refuse a call that has its memory.
static cudaError_t taken(cudaError_t e) {
    if (e == cudaErrorMemoryAllocation) cudaGetLastError();
    return e;
}

cudaError_t dev_malloc(void** p, size_t bytes) {
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    return taken(cudaMalloc(p, bytes));
}

cudaError_t dev_alloc(void** p, size_t bytes, cudaStream_t st) {
    std::call_once(g_pool_once, [] {
        // Keep freed blocks in this process's default pool so that repeated
        // graph/sketch builds do not return memory to the CUDA driver and map it
        // again. The attribute belongs to this process's pool only.
        int dev = 0;
        cudaMemPool_t pool;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
            uint64_t thr = UINT64_MAX;
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
        }
    });
    *p = nullptr;
    if (bytes == 0) bytes = 16;
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    return taken(cudaMallocAsync(p, bytes, st));
}

void dev_free(void* p, cudaStream_t st) {
    if (p) cudaFreeAsync(p, st);
}

void dev_trim(cudaStream_t st) {
    int dev = 0;
    cudaMemPool_t pool;
    if (cudaStreamSynchronize(st) == cudaSuccess && cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess)
        cudaMemPoolTrimTo(pool, 0);
}

int sm_count() {
    static int cached = 0;
    if (cached == 0) {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        cached = v > 0 ? v : 1;
    }
    return cached;
}

// ------------------------------------------------------------------- scan
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint64_t shfl_up_t(uint64_t v, int d) { return __shfl_up_sync(kFull, v, d); }
__device__ __forceinline__ u128 shfl_up_t(u128 v, int d) {
    uint64_t lo = (uint64_t)v, hi = (uint64_t)(v >> 64);
    lo = __shfl_up_sync(kFull, lo, d);
    hi = __shfl_up_sync(kFull, hi, d);
    return ((u128)hi << 64) | lo;
}

// Exclusive scan of one value per thread across the block; returns the
// thread's exclusive prefix, and the block total in *total.
template <typename T>
__device__ T block_exclusive_scan(T val, T* total) {
    __shared__ T s_warp[kScanThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T incl = val;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T y = shfl_up_t(incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) s_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        T w = lane < kScanThreads / 32 ? s_warp[lane] : T(0);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            T y = shfl_up_t(w, d);
            if (lane >= d) w += y;
        }
        if (lane < kScanThreads / 32) s_warp[lane] = w;
    }
    __syncthreads();
    const T warp_excl = wid > 0 ? s_warp[wid - 1] : T(0);
    *total = s_warp[kScanThreads / 32 - 1];
    __syncthreads();
    return warp_excl + incl - val;
}

template <typename TIn, typename T>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const TIn* __restrict__ in, int64_t n,
                                                              T* __restrict__ partial) {
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
        if (base + k < n) s += (T)in[base + k];
    T tot;
    block_exclusive_scan<T>(s, &tot);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

template <typename TIn, typename T>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const TIn* __restrict__ in, int64_t n,
                                                             const T* __restrict__ offsets,
                                                             T* __restrict__ out) {
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    T v[kScanItems];
    T s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = (base + k < n) ? (T)in[base + k] : T(0);
        s += v[k];
    }
    T tot;
    T run = block_exclusive_scan<T>(s, &tot) + (offsets ? offsets[blockIdx.x] : T(0));
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) out[n] = run;
}

template <typename TIn, typename T>
static cudaError_t scan_impl(const TIn* in, T* out, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaMemsetAsync(out, 0, sizeof(T), st);
    const int64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb == 1) {
        k_scan_apply<TIn, T><<<1, kScanThreads, 0, st>>>(in, n, (const T*)nullptr, out); note_launch();
        return cudaGetLastError();
    }
    T* partial = nullptr;
    T* pscan = nullptr;
    cudaError_t e = dev_alloc_t(&partial, (size_t)nb, st);
    if (e != cudaSuccess) return e;
    e = dev_alloc_t(&pscan, (size_t)nb + 1, st);
    if (e != cudaSuccess) { dev_free(partial, st); return e; }
    k_scan_reduce<TIn, T><<<(unsigned)nb, kScanThreads, 0, st>>>(in, n, partial); note_launch();
    e = scan_impl<T, T>(partial, pscan, nb, st);
    if (e == cudaSuccess) {
        k_scan_apply<TIn, T><<<(unsigned)nb, kScanThreads, 0, st>>>(in, n, pscan, out); note_launch();
        e = cudaGetLastError();
    }
    dev_free(partial, st);
    dev_free(pscan, st);
    return e;
}

cudaError_t scan_u32_to_u64(const uint32_t* in, uint64_t* out, int64_t n, cudaStream_t st) {
    return scan_impl<uint32_t, uint64_t>(in, out, n, st);
}
cudaError_t scan_u64(const uint64_t* in, uint64_t* out, int64_t n, cudaStream_t st) {
    return scan_impl<uint64_t, uint64_t>(in, out, n, st);
}
cudaError_t scan_u128(const u128* in, u128* out, int64_t n, cudaStream_t st) {
    return scan_impl<u128, u128>(in, out, n, st);
}

// ------------------------------------------------------------- edge sort
// Stable LSD radix sort of the edges by key dst << src_bits | src, the input
// index as value (so equal keys keep input order), in 8-bit digits. One
// kernel reads the edges once and counts every digit of every pass; then one
// kernel a pass ("onesweep"): each CTA claims the next tile from a ticket,
// ranks its items per warp (one vote a digit bit, warp-striped loads: positions
// in warp order, so the ranking is stable), publishes the tile's per-digit
// counts, lays the tile out in shared memory in digit order, looks back over
// the previous tiles' published counts for its global offsets (decoupled
// look-back), and writes the tile out, so that each digit's items leave as a
// contiguous run. The first pass builds the keys from the edge arrays in
// registers.
// A pass is bound by instruction issue (the votes: 0.7 of the ALU pipe) and by
// the look-back's latency, at about half of the copy bandwidth. 7 10^7 edges,
// 44-bit keys in five passes, whole graph load: 5.71 ms with match_any ranks
// and tiles of 4096 items on 256 threads, 4.46 with votes and 6144 items on
// 512 threads, two CTAs an SM (4096 items, three CTAs: 4.7; 7168: 4.6; 8192 on
// one CTA: 6.4); 1.4 10^8 edges 10.7 -> 8.2 ms.
constexpr int kOsThreads = 512;
constexpr int kOsItems = 12;
constexpr int kOsGroup = 4;                     // of a thread's items ranked at a time
constexpr int kOsTile = kOsThreads * kOsItems;  // 6144 items
constexpr int kOsWarps = kOsThreads / 32;
constexpr int kOsMaxPasses = 8;
// status word of (tile, digit): state in bits 62-63 (1: the tile's own
// count, 2: inclusive prefix over tiles 0 .. tile), the pass tag (pass + 1)
// in bits 56-61, the count in bits 0-55. Words of another pass read as not
// yet published, so one zeroing serves every pass.
constexpr unsigned long long kOsAgg = 1ull << 62, kOsIncl = 2ull << 62;
constexpr unsigned long long kOsCount = (1ull << 56) - 1;
constexpr uint32_t kOsSpinLimit = 1u << 22;  // polls of one word before giving up (~0.3 s)
constexpr int kOsWindow = 8;                 // predecessor tiles read at once in the look-back

__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint64_t edge_key(const int32_t* src, const int32_t* dst, int64_t e, int src_bits) {
    return ((uint64_t)(uint32_t)dst[e] << src_bits) | (uint64_t)(uint32_t)src[e];
}

// Pass p sorts on the digit (key >> shift[p]) & (2^bits[p] - 1), bits[p] in
// {8, 9}: a 9-bit pass has 512 digits, two a thread in the per-digit steps,
// so that 50- and 52-bit keys take six passes instead of seven.
constexpr int kOsMaxDigits = 512;
struct OsPasses {
    int n;
    int shift[kOsMaxPasses];
    int bits[kOsMaxPasses];
};

// Digit counts of every pass: hist[p * kOsMaxDigits + d] = #{edges whose key
// has digit d in pass p}.
__global__ void __launch_bounds__(256) k_os_hist(const int32_t* __restrict__ src, const int32_t* __restrict__ dst,
                                                 int64_t m, int src_bits, OsPasses ps,
                                                 unsigned long long* __restrict__ hist) {
    __shared__ uint32_t s_h[kOsMaxPasses * kOsMaxDigits];
    for (int i = threadIdx.x; i < ps.n * kOsMaxDigits; i += 256) s_h[i] = 0;
    __syncthreads();
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = edge_key(src, dst, e, src_bits);
#pragma unroll
        for (int p = 0; p < kOsMaxPasses; ++p)  // static indices: the pass table stays in the parameters
            if (p < ps.n)
                atomicAdd(&s_h[p * kOsMaxDigits + (uint32_t)((key >> ps.shift[p]) & ((1u << ps.bits[p]) - 1u))], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ps.n * kOsMaxDigits; i += 256)
        if (s_h[i]) atomicAdd(&hist[i], (unsigned long long)s_h[i]);
}

// Exclusive prefix of each pass's digit counts, in place: base[p * kOsMaxDigits + d].
// A block a pass, by warp scans (a thread summing its predecessors one by one,
// pass after pass, took 12-16 us of a small load).
__global__ void __launch_bounds__(kOsMaxDigits) k_os_bases(unsigned long long* __restrict__ hist) {
    __shared__ unsigned long long s_w[kOsMaxDigits / 32];
    unsigned long long* const h = hist + blockIdx.x * kOsMaxDigits;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned long long c = h[threadIdx.x];
    unsigned long long x = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    unsigned long long before = lane < wid ? s_w[lane] : 0;  // lane < wid < kOsMaxDigits / 32 <= 32
    static_assert(kOsMaxDigits / 32 <= 32, "a lane a warp");
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(kFull, before, d);
    h[threadIdx.x] = before + x - c;
}

// One pass on the kBits-bit digit at `shift`. kFirst: the items are the
// edges (key built from src / dst, value = input index). kLast: the sorted
// items leave as the CSR arrays (source = the key's low src_bits bits,
// destination = the rest, input index) instead of keys and values. Dynamic
// shared memory: kOsTile keys and values.
struct OsOut {
    uint64_t* keys;
    uint32_t* vals;
    int32_t* csr_src;
    uint32_t* csr_dst;
    uint32_t* perm;
};

template <bool kFirst, bool kLast, int kBits>
__global__ void __launch_bounds__(kOsThreads, 2) k_os_pass(
    const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int src_bits,
    const uint64_t* __restrict__ keys_in, const uint32_t* __restrict__ vals_in, OsOut out, int64_t n, int shift,
    unsigned long long tag,
    const unsigned long long* __restrict__ base, unsigned long long* __restrict__ status,
    unsigned int* __restrict__ ticket, unsigned int* __restrict__ gave_up) {
    constexpr int kDigits = 1 << kBits;  // thread t < kDigits owns digit t
    constexpr uint32_t kMask = kDigits - 1;
    static_assert(kDigits <= kOsThreads && kOsTile <= 65536, "a digit a thread; positions in the tile fit 16 bits");
    extern __shared__ __align__(16) unsigned char os_smem[];
    uint64_t* s_keys = reinterpret_cast<uint64_t*>(os_smem);
    uint32_t* s_vals = reinterpret_cast<uint32_t*>(s_keys + kOsTile);
    // per warp: digit counts, then the tile position of the warp's first (16 bits each, two a word)
    __shared__ uint32_t s_wcnt[kOsWarps][kDigits / 2];
    __shared__ uint32_t s_out[kDigits];  // output position of a digit's items less their tile position
    __shared__ uint32_t s_wsum[kOsWarps];
    __shared__ uint32_t s_tile, s_bad;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool owner = tid < kDigits;
    uint16_t* const my_cnt = reinterpret_cast<uint16_t*>(&s_wcnt[0][0]) + tid;  // + w kDigits: warp w's
    if (tid == 0) {
        s_tile = atomicAdd(ticket, 1u);
        s_bad = 0;
    }
    const unsigned long long digit_base = owner ? base[tid] : 0;  // in flight while the tile loads
    for (int i = tid; i < kOsWarps * kDigits / 2; i += kOsThreads) (&s_wcnt[0][0])[i] = 0;
    __syncthreads();
    const uint32_t tile = s_tile;
    const int64_t t0 = (int64_t)tile * kOsTile;
    const int64_t wb = t0 + (int64_t)wid * (32 * kOsItems) + lane;  // this lane's items: wb + 32 c
    const int left = (int)max((int64_t)0, min((int64_t)(32 * kOsItems), n - wb));  // item c is there if 32 c < left
    uint64_t key[kOsItems];
#pragma unroll
    for (int c = 0; c < kOsItems; ++c) {
        key[c] = 0;
        if (32 * c < left) key[c] = kFirst ? edge_key(src, dst, wb + 32 * c, src_bits) : keys_in[wb + 32 * c];
    }
    // rank within the warp: earlier chunks, then lower lanes. The lanes with a
    // lane's digit by one vote a bit (a match instruction is slower); then the
    // counter updates in chunk order, none waiting for the one before, and the
    // broadcasts, kOsGroup of each in flight
    uint32_t rnk[kOsItems];  // digit << 16 | rank
#pragma unroll
    for (int g = 0; g < kOsItems; g += kOsGroup) {
        uint32_t peers[kOsGroup], old[kOsGroup];
#pragma unroll
        for (int q = 0; q < kOsGroup; ++q) {
            const int c = g + q;
            const uint32_t d = (uint32_t)(key[c] >> shift) & kMask;
            rnk[c] = d << 16;
            peers[q] = __ballot_sync(kFull, 32 * c < left);
#pragma unroll
            for (int b = 0; b < kBits; ++b) {
                const uint32_t ones = __ballot_sync(kFull, (d >> b) & 1u);
                const uint32_t mine = (uint32_t)((int32_t)(d << (31 - b)) >> 31);  // all bits as the lane's bit b
                peers[q] &= ~(ones ^ mine);
            }
            old[q] = 0;
            if (32 * c < left && (peers[q] & lanemask_lt()) == 0)
                old[q] = atomicAdd(&s_wcnt[wid][d >> 1], (uint32_t)__popc(peers[q]) << (16 * (d & 1u)));
            __syncwarp();  // this chunk's counts come before the next chunk's
        }
#pragma unroll
        for (int q = 0; q < kOsGroup; ++q) {
            const uint32_t d = rnk[g + q] >> 16;
            const uint32_t before = __shfl_sync(kFull, old[q], __ffs(peers[q]) - 1) >> (16 * (d & 1u));
            rnk[g + q] += (before & 0xFFFFu) + (uint32_t)__popc(peers[q] & lanemask_lt());
        }
    }
    uint32_t val[kOsItems];  // arrive while the counts are scanned
#pragma unroll
    for (int c = 0; c < kOsItems; ++c) {
        val[c] = 0;
        if (32 * c < left) val[c] = kFirst ? (uint32_t)(wb + 32 * c) : vals_in[wb + 32 * c];
    }
    __syncthreads();
    // the owned digit's count in the tile, published at once
    uint32_t cnt = 0;
    if (owner) {
#pragma unroll
        for (int w = 0; w < kOsWarps; ++w) cnt += my_cnt[w * kDigits];
        st_relaxed_u64(status + (size_t)tile * kDigits + tid, (tile == 0 ? kOsIncl : kOsAgg) | tag | cnt);
    }
    // tile-local digit starts: exclusive scan of the counts in digit order, and
    // from them each warp's start in the digit
    uint32_t start = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t z = __shfl_up_sync(kFull, start, o);
        if (lane >= o) start += z;
    }
    if (lane == 31) s_wsum[wid] = start;
    __syncthreads();
    start -= cnt;
    for (int w = 0; w < wid; ++w) start += s_wsum[w];
    if (owner) {
        uint32_t run = start;
#pragma unroll
        for (int w = 0; w < kOsWarps; ++w) {
            const uint32_t c2 = my_cnt[w * kDigits];
            my_cnt[w * kDigits] = (uint16_t)run;
            run += c2;
        }
    }
    __syncthreads();
    // the tile in shared memory in digit order
#pragma unroll
    for (int c = 0; c < kOsItems; ++c) {
        if (32 * c < left) {
            const uint32_t pos = reinterpret_cast<const uint16_t*>(s_wcnt[wid])[rnk[c] >> 16] + (rnk[c] & 0xFFFFu);
            s_keys[pos] = key[c];
            s_vals[pos] = val[c];
        }
    }
    // (the keys' registers are free, and the earlier tiles have had the placement's
    // time to publish) look back over them for the owned digit's items before the
    // tile, kOsWindow tiles a read: sum their own counts back to the first
    // inclusive prefix, waiting on the first tile not yet published
    if (owner) {
        unsigned long long excl = 0;
        int64_t t = (int64_t)tile - 1;  // the next tile to account for
        uint32_t spins = 0;
        bool done = tile == 0;
        while (!done) {
            unsigned long long v[kOsWindow];
#pragma unroll
            for (int k = 0; k < kOsWindow; ++k)
                v[k] = t - k >= 0 ? ld_relaxed_u64(status + (size_t)(t - k) * kDigits + tid) : 0;
            int k = 0;
#pragma unroll
            for (int q = 0; q < kOsWindow; ++q) {
                const bool ready = (v[q] & (63ull << 56)) == tag && (v[q] >> 62) != 0;
                if (!ready) break;
                excl += v[q] & kOsCount;
                ++k;
                if ((v[q] >> 62) == 2) {
                    done = true;
                    break;
                }
            }
            if (done) break;
            t -= k;  // tile 0 is always inclusive, so t stays >= 0
            if (k < kOsWindow) {  // tile t is not published yet
                if (++spins > kOsSpinLimit) {  // cannot happen while every claimed tile runs; never hang
                    atomicOr(gave_up, 1u);
                    s_bad = 1;
                    break;
                }
                __nanosleep(32);
            }
        }
        if (tile > 0)
            st_relaxed_u64(status + (size_t)tile * kDigits + tid, kOsIncl | tag | ((excl + cnt) & kOsCount));
        s_out[tid] = (uint32_t)(digit_base + excl) - start;  // positions are below 2^32
    }
    __syncthreads();
    if (s_bad) return;  // offsets unknown: write nothing (the host reports the failure)
    const int tile_n = (int)min((int64_t)kOsTile, n - t0);
    for (int i = tid; i < tile_n; i += kOsThreads) {
        const uint64_t k = s_keys[i];
        const uint32_t g = s_out[(uint32_t)((k >> shift) & kMask)] + (uint32_t)i;
        if ((int64_t)g >= n) {  // inconsistent counts (cannot happen): never write out of bounds
            atomicOr(gave_up, 2u);
            continue;
        }
        if (kLast) {
            out.csr_src[g] = (int32_t)(k & ((1ull << src_bits) - 1));
            out.csr_dst[g] = (uint32_t)(k >> src_bits);
            out.perm[g] = s_vals[i];
        } else {
            out.keys[g] = k;
            out.vals[g] = s_vals[i];
        }
    }
}

// The passes for keys of `bits` bits: P = ceil(bits / 9) passes (at least
// one), the last max(0, bits - 8 P) of them 9 bits wide, the others 8 (50
// bits: 8, 8, 8, 8, 9, 9; 40 bits: five of 8).
static OsPasses os_passes(int bits) {
    OsPasses ps{};
    const int P = std::max(1, (bits + 8) / 9);
    const int nine = std::max(0, bits - 8 * P);  // <= P, as 9 P >= bits
    ps.n = P;
    int sh = 0;
    for (int p = 0; p < P; ++p) {
        ps.bits[p] = p >= P - nine ? 9 : 8;
        ps.shift[p] = sh;
        sh += ps.bits[p];
    }
    return ps;
}

template <int kBits>
static cudaError_t os_pass_attr(size_t smem) {
    const void* fns[4] = {(const void*)k_os_pass<true, false, kBits>, (const void*)k_os_pass<false, false, kBits>,
                          (const void*)k_os_pass<true, true, kBits>, (const void*)k_os_pass<false, true, kBits>};
    for (const void* f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int kBits, bool kLast>
static void os_launch(bool first, int64_t ntiles, size_t smem, cudaStream_t st, const int32_t* src, const int32_t* dst,
                      int src_bits, const uint64_t* ksrc, const uint32_t* vsrc, const OsOut& out, int64_t m, int shift,
                      unsigned long long tag, const unsigned long long* base, unsigned long long* status,
                      unsigned int* ticket, unsigned int* gave_up) {
    if (first)
        k_os_pass<true, kLast, kBits><<<(unsigned)ntiles, kOsThreads, smem, st>>>(
            src, dst, src_bits, nullptr, nullptr, out, m, shift, tag, base, status, ticket, gave_up);
    else
        k_os_pass<false, kLast, kBits><<<(unsigned)ntiles, kOsThreads, smem, st>>>(
            nullptr, nullptr, src_bits, ksrc, vsrc, out, m, shift, tag, base, status, ticket, gave_up);
}

cudaError_t sort_edges(const int32_t* src, const int32_t* dst, int64_t m, int src_bits, int32_t* csr_src,
                       uint32_t* csr_dst, uint32_t* perm, uint64_t* keys_a, uint32_t* vals_a, uint64_t* keys_b,
                       uint32_t* vals_b, unsigned int* gave_up, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    const OsPasses ps = os_passes(2 * src_bits);
    if (ps.n > kOsMaxPasses) return cudaErrorInvalidValue;
    const int passes = ps.n;
    const int64_t ntiles = (m + kOsTile - 1) / kOsTile;
    const size_t smem = (size_t)kOsTile * (sizeof(uint64_t) + sizeof(uint32_t));
    // set on every call: the attribute belongs to the current device
    cudaError_t attr_err = os_pass_attr<8>(smem);
    if (attr_err == cudaSuccess) attr_err = os_pass_attr<9>(smem);
    if (attr_err != cudaSuccess) return attr_err;
    unsigned long long *hist = nullptr, *status = nullptr;
    unsigned int* tickets = nullptr;
    // one allocation, zeroed at once: the digit counts, the status words, the tickets
    const size_t words = (size_t)(passes + ntiles) * kOsMaxDigits + (size_t)passes;
    cudaError_t e = dev_alloc_t(&hist, words, st);
    if (e == cudaSuccess) {
        status = hist + (size_t)passes * kOsMaxDigits;
        tickets = reinterpret_cast<unsigned int*>(status + (size_t)ntiles * kOsMaxDigits);
        e = cudaMemsetAsync(hist, 0, words * sizeof(unsigned long long), st);
    }
    if (e == cudaSuccess) {
        const int grid = (int)std::min<int64_t>((int64_t)sm_count() * 8, std::max<int64_t>(1, (m + 255) / 256));
        k_os_hist<<<grid, 256, 0, st>>>(src, dst, m, src_bits, ps, hist); note_launch();
        k_os_bases<<<passes, kOsMaxDigits, 0, st>>>(hist); note_launch();
        e = cudaGetLastError();
    }
    const uint64_t* ksrc = nullptr;
    const uint32_t* vsrc = nullptr;
    for (int p = 0; p < passes && e == cudaSuccess; ++p) {
        // passes alternate between the a and b buffers; the last one writes the CSR arrays
        const bool last = p == passes - 1;
        const OsOut out{p % 2 == 0 ? keys_a : keys_b, p % 2 == 0 ? vals_a : vals_b, csr_src, csr_dst, perm};
        const unsigned long long tag = (unsigned long long)(p + 1) << 56;
        const unsigned long long* base = hist + p * kOsMaxDigits;
        if (ps.bits[p] == 9) {
            if (last)
                os_launch<9, true>(p == 0, ntiles, smem, st, src, dst, src_bits, ksrc, vsrc, out, m, ps.shift[p], tag,
                                   base, status, tickets + p, gave_up);
            else
                os_launch<9, false>(p == 0, ntiles, smem, st, src, dst, src_bits, ksrc, vsrc, out, m, ps.shift[p], tag,
                                    base, status, tickets + p, gave_up);
        } else {
            if (last)
                os_launch<8, true>(p == 0, ntiles, smem, st, src, dst, src_bits, ksrc, vsrc, out, m, ps.shift[p], tag,
                                   base, status, tickets + p, gave_up);
            else
                os_launch<8, false>(p == 0, ntiles, smem, st, src, dst, src_bits, ksrc, vsrc, out, m, ps.shift[p], tag,
                                    base, status, tickets + p, gave_up);
        }
        note_launch();
        e = cudaGetLastError();
        ksrc = out.keys;
        vsrc = out.vals;
    }
    dev_free(hist, st);
    return e;
}

// -------------------------------------------------------------------- sum
__global__ void k_sum_u64(const uint64_t* __restrict__ in, int64_t n, unsigned long long* out) {
    unsigned long long s = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s += in[i];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(kFull, s, d);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

cudaError_t sum_u64(const uint64_t* in, int64_t n, unsigned long long* out, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    int blocks = (int)std::min<int64_t>((int64_t)sm_count() * 4, std::max<int64_t>(1, (n + 255) / 256));
    k_sum_u64<<<blocks, 256, 0, st>>>(in, n, out); note_launch();
    return cudaGetLastError();
}

}  // namespace skis
