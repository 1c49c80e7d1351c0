"""The coverage scan of small sketches under any order of its threads that CUDA's model allows, on the host: a warp's threads may run ahead of
one another up to the next collective, and votes and shuffles order no memory."""
import subprocess

import pytest

import warp_emu

COVER = r"""
//KERNELS//
int main(int argc, char** argv) {
    const unsigned seed = atoi(argv[1]);
    const int glog = atoi(argv[2]);
    const uint64_t T = 77;
    std::mt19937 rng(seed);
    std::vector<uint64_t> off(T), qmask(50);
    std::vector<uint32_t> len(T);
    std::vector<int32_t> arena;
    for (auto& x : qmask) x = rng() % 3 ? 0 : (uint64_t)rng() << (rng() % 32) & (uint64_t)rng() << (rng() % 32);
    std::vector<unsigned long long> cov(64, 0), want(64, 0);
    for (uint64_t j = 0; j < T; ++j) {
        off[j] = arena.size();
        len[j] = rng() % 40;
        uint64_t m = 0;
        for (uint32_t i = 0; i < len[j]; ++i) {
            arena.push_back(rng() % 50);
            m |= qmask[arena.back()];
        }
        for (int b = 0; b < 64; ++b) want[b] += m >> b & 1;
    }
    emu::defer_or = true;
    emu::run(kCovThreads, 0, 1, seed, [&] {
        k_coverage(off.data(), len.data(), T, arena.data(), qmask.data(), nullptr, 0, glog, cov.data());
    });
    return cov == want ? 0 : 1;
}
"""


@pytest.mark.parametrize("glog", [0, 3, 5])
def test_coverage_reads_a_sample_s_queries_after_every_lane_has_added_its_own(tmp_path, glog):
    exe = warp_emu.build(tmp_path, "cover.cu", ["kCovThreads", "kCovBlocks", "warp_members", "kFilterLog2", "filter_index",
                                                "k_coverage"], COVER)
    for seed in range(8):
        assert subprocess.run([exe, str(seed), str(glog)], timeout=120).returncode == 0
