"""The coverage scan in sample order under any order of its threads that CUDA's model allows, on the host: a warp's threads may run ahead of
one another up to the next collective, and votes and shuffles order no memory."""
import subprocess

import pytest

import warp_emu

SCAN = r"""
static inline void prefetch_l2(const void*, uint32_t) {}
alignas(16) uint32_t s_f[1 << 15];
//KERNELS//
// T samples of len members each, every `gap`-th member a seed of query 0
int main(int argc, char** argv) {
    const unsigned seed = atoi(argv[1]);
    const uint64_t T = atoi(argv[2]), len = atoi(argv[3]), gap = atoi(argv[4]);
    const unsigned long long cap = atoi(argv[5]);
    std::vector<uint64_t> off(T), qmask(64, 0);
    std::vector<uint32_t> hl(T, (uint32_t)len), qbits(2, 0), touched(T);
    int32_t* const arena = (int32_t*)aligned_alloc(16, (T * len + 4) * 4);
    uint64_t want = 0;
    for (uint64_t j = 0; j < T; ++j) {
        off[j] = j * len;
        bool hit = false;
        for (uint64_t i = 0; i < len; ++i) {
            arena[j * len + i] = (j * len + i) % gap == 0 ? 7 : 9;
            hit = hit || arena[j * len + i] == 7;
        }
        want += hit;
    }
    qbits[0] = 1u << 7;
    qmask[7] = 1;
    std::vector<unsigned long long> smask(T, 0), cov(64, 0), hits(1 << 16, 0);
    unsigned long long ntouched = 0, cursor = 0, nhits = 0;
    emu::run(kScanThreads, 0, 1, seed, [&] {
        k_scan_ordered(off.data(), hl.data(), T, 10, arena, qbits.data(), 2, 0, qmask.data(), smask.data(), touched.data(),
                       &ntouched, &cursor, hits.data(), &nhits, cap, cov.data());
    });
    emu::run(256, 0, 1, seed, [&] {
        k_scan_hits(hits.data(), &nhits, cap, off.data(), T, 10, arena, qmask.data(), smask.data(), touched.data(),
                    &ntouched, cov.data());
    });
    fprintf(stderr, "%llu samples covered, %llu are\n", cov[0], (unsigned long long)want);
    return cov[0] == want && ntouched == want ? 0 : 1;
}
"""
SCAN_NAMES = ["kScanThreads", "kScanUnroll", "kScanHits", "kScanMembers", "kScanAhead", "kFilterLog2", "filter_index",
              "k_scan_ordered", "k_scan_hits"]


@pytest.fixture(scope="module")
def scan(tmp_path_factory):
    return warp_emu.build(tmp_path_factory.mktemp("scan"), "cover.cu", SCAN_NAMES, SCAN)


# a warp step tests 512 members: 8 to 9 steps to the 64 hits at which a warp's hits join the list, 1, and 2; with a
# list that holds all of them, and one that is full
@pytest.mark.parametrize("gap", [65, 8, 11])
@pytest.mark.parametrize("cap", [1 << 16, 5])
def test_ordered_scan_counts_whatever_lane_runs_ahead(scan, gap, cap):
    for seed in range(4):
        r = subprocess.run([scan, str(seed), "1500", "9", str(gap), str(cap)], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stderr
