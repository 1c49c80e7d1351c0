"""The index walk's queue of a long list's chunks, for a seed whose place in its batch needs more than 32 bits (64 queries
of a graph of 2^27 vertices can hold 2^33 seeds): the block that such a seed falls to, on the host (the kernel's own text),
with only that seed in memory."""
import subprocess

import pytest

import warp_emu

DRIVER = r"""
struct skis_sketch;
//KERNELS//
int main(int argc, char** argv) {
    const uint64_t at = strtoull(argv[1], 0, 10);  // the seed's place: a multiple of 8
    const uint64_t len = strtoull(argv[2], 0, 10), cap = strtoull(argv[3], 0, 10);
    const int32_t seeds[8] = {1, 0, 0, 0, 0, 0, 0, 0};  // lists of vertex 1: len entries, vertex 0: one
    const int64_t off[3] = {0, (int64_t)at, (int64_t)at + 8};
    const uint64_t inv_off[3] = {0, 1, 1 + len};
    std::vector<uint32_t> inv(1 + len);
    inv[0] = (uint32_t)len;
    for (uint64_t x = 0; x < len; ++x) inv[1 + x] = (uint32_t)x;
    std::vector<unsigned long long> smask(len + 1, 0), cov(65, 0);
    std::vector<uint64_t> queue(cap, ~0ull);
    InvWalk a;
    a.off = off;
    a.seeds = seeds - at;
    a.q0 = 0;
    a.qn = 2;
    a.seed_base = 0;
    a.nseeds = at + 8;
    a.n = 2;
    a.inv_off = inv_off;
    a.inv = inv.data();
    a.smask = smask.data();
    a.cov = cov.data();
    a.queue = queue.data();
    a.queue_cap = cap;
    a.nqueue = cov.data() + 64;
    for (int mode = 0; mode < 3; ++mode) {
        // the queue's items go to the grid's first warps
        emu::run(kCovThreads, at / 8, at / 8 + 1, 7, [&] { k_cover_inv(a, mode); });
        if (at && mode) {
            InvWalk b = a;
            b.nseeds = 0;
            emu::run(kCovThreads, 0, 1, 7, [&] { k_cover_inv(b, mode); });
        }
    }
    for (auto m : smask)
        if (m) return 2;
    fprintf(stderr, "%llu %llu\n", cov[0], cov[1]);
    return cov[0] == 0 && cov[1] == len + 1 ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    return warp_emu.build(tmp_path_factory.mktemp("inv"), "cover.cu",
                          ["kCovThreads", "kInvChunk", "kInvChunkBits", "InvWalk", "walk_list", "k_cover_inv"], DRIVER)


@pytest.mark.parametrize("at", [0, 8, 1 << 31, 1 << 32, (1 << 33) + 800])
@pytest.mark.parametrize("length,cap", [(256, 100), (257, 100), (900, 100), (900, 2), (5000, 100)])
def test_chunks_of_a_seed_at_any_place(exe, at, length, cap):
    r = subprocess.run([exe, str(at), str(length), str(cap)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stderr)
