"""``k_greedy_rounds`` on the host (warp_emu): one block of it over a random sketch, with grid barriers that the driver
stands in for."""
import warp_emu

NAMES = ["kHotBits", "kHotSlots", "kHotEmpty", "sub_merged", "Cand", "kNone", "no_cand", "cand_better", "warp_best_lane",
         "ldcg_cand", "GreedyCtl", "GreedyArgs", "kGreedyThreads", "kGreedySegLog", "kGreedySeg", "kBuckets", "kPoolMin",
         "kSegRounds", "greedy_bucket", "k_greedy_init", "k_greedy_rounds"]

DRIVER = r"""
struct GreedyCtl;
static int barriers_left = 1 << 30;       // grid barriers before one runs out
static std::function<void()> other_blocks;  // what they have written when a barrier is reached
struct GridBar {
    GreedyCtl* ctl;
    uint32_t* failed;
    uint32_t goal;
    void arrive(bool) { ++goal; }
    bool wait(bool) {
        if (threadIdx.x == 0) {
            if (barriers_left-- == 0) *failed = 1;
            else if (other_blocks) other_blocks();
        }
        __syncthreads();
        return *failed == 0;
    }
    bool sync() {
        __syncthreads();
        arrive(true);
        return wait(true);
    }
};
static double u128_to_double(u128 v) { return (double)v; }
//KERNELS//
// n elements, whatever follows them unreadable
template <class T>
static T* guarded(size_t n) {
    const size_t page = 4096, bytes = (n * sizeof(T) + 15 + page - 1) / page * page;
    char* p = (char*)mmap(nullptr, bytes + (1ull << 36), PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (p == (char*)MAP_FAILED) abort();
    mprotect(p, bytes, PROT_READ | PROT_WRITE);
    return (T*)(p + bytes - (n * sizeof(T) + 15) / 16 * 16);
}
struct Sketch {
    GreedyArgs a;
    std::vector<std::vector<uint32_t>> members;
    int64_t n;
    uint64_t T;
    // T samples of `size` members; blocks the grid would have
    Sketch(int64_t n_, uint64_t T_, int size, int32_t k, unsigned blocks, unsigned seed) : n(n_), T(T_) {
        std::mt19937 rng(seed);
        std::vector<std::vector<uint32_t>> lists(n);
        uint64_t* h_off = guarded<uint64_t>(T);
        uint32_t* h_len = guarded<uint32_t>(T);
        int32_t* arena = guarded<int32_t>(T * size);
        uint64_t at = 0;
        for (uint64_t j = 0; j < T; ++j) {
            std::vector<uint32_t> m;
            while ((int)m.size() < size) {
                const uint32_t u = (uint32_t)(n * (double)(rng() % 65536) / 65536 * (rng() % 65536) / 65536);
                if (std::find(m.begin(), m.end(), u) == m.end()) m.push_back(u);
            }
            h_off[j] = at;
            h_len[j] = size;
            for (uint32_t u : m) {
                arena[at++] = (int32_t)u;
                lists[u].push_back((uint32_t)j);
            }
            members.push_back(m);
        }
        uint64_t* inv_off = guarded<uint64_t>(n + 1);
        uint32_t* inv = guarded<uint32_t>(at);
        uint64_t* w = guarded<uint64_t>(n);
        uint64_t x = 0, W = 0;
        for (int64_t v = 0; v < n; ++v) {
            inv_off[v] = x;
            for (uint32_t j : lists[v]) inv[x++] = j;
            W += w[v] = 1 + rng() % ((1u << 20) - 1);
        }
        inv_off[n] = x;
        a.w = w;
        a.inS = guarded<uint8_t>(n + 16);
        a.delta = guarded<uint32_t>(n);
        a.n = n;
        a.W = W;
        a.T = T;
        a.ratio = (double)T / (double)W;
        a.f = 20;
        a.k = k;
        a.inv_off = inv_off;
        a.inv = inv;
        a.h_off = h_off;
        a.h_len = h_len;
        a.arena = arena;
        a.covered = guarded<uint32_t>((T + 31) / 32);
        a.nseg = (n + kGreedySeg - 1) / kGreedySeg;
        a.partial = guarded<Cand>(blocks);
        a.seg_best = guarded<Cand>(a.nseg);
        a.pool = guarded<uint32_t>(kGreedyThreads);
        a.hist = guarded<uint32_t>(kBuckets);
        a.ctl = guarded<GreedyCtl>(1);
        a.seeds = guarded<int32_t>(k);
        a.cov_out = guarded<int64_t>(k);
        a.est_out = guarded<double>(k);
        a.ris = 0;
        memset(a.partial, 0xFF, blocks * sizeof(Cand));  // what an allocation may hold
        memset(a.pool, 0xFF, kGreedyThreads * sizeof(uint32_t));
        emu::run(kGreedyThreads, 0, 1, seed, [&] { k_greedy_init(a); });
    }
    bool right() const {  // the seeds are plain greedy's
        std::vector<char> covered(T, 0), in(n, 0);
        for (int32_t r = 0; r < a.k; ++r) {
            std::vector<uint64_t> d(n, 0);
            for (uint64_t j = 0; j < T; ++j)
                if (!covered[j])
                    for (uint32_t u : members[j]) ++d[u];
            int64_t best = -1;
            u128 key = 0;
            for (int64_t v = 0; v < n; ++v) {
                const u128 x = (u128)d[v] * a.W + (u128)T * ((1ull << a.f) - a.w[v]);
                if (!in[v] && (best < 0 || x > key)) best = v, key = x;
            }
            if (a.seeds[r] != best) {
                fprintf(stderr, "seed %d is %d, not %lld\n", r, a.seeds[r], (long long)best);
                return false;
            }
            in[best] = 1;
            for (uint64_t j = 0; j < T; ++j)
                for (uint32_t u : members[j])
                    if (u == best) covered[j] = 1;
        }
        return true;
    }
};
"""


def build(tmp_path, main):
    return warp_emu.build(tmp_path, "cover.cu", NAMES, DRIVER + main)
