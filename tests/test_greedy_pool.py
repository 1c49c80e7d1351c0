"""Greedy's candidate pool filled by a histogram that promises room for fewer vertices than reach the cut (as when the two
places that round a key to its bucket would round differently): a vertex that finds the pool full still counts as one of
the others, so the seeds are plain greedy's. On the host (the kernel's own text)."""
import subprocess

import pytest

import greedy_emu

MAIN = r"""
int main(int argc, char** argv) {
    const unsigned seed = atoi(argv[1]);
    const uint32_t missing = atoi(argv[2]);
    Sketch s(1500, 200, 20, 6, 1, seed);
    uint32_t left = missing;  // the histogram's best vertices are not counted
    for (int i = kBuckets - 1; i >= 0 && left; --i) {
        const uint32_t c = std::min(s.a.hist[i], left);
        s.a.hist[i] -= c;
        left -= c;
    }
    emu::run(kGreedyThreads, 0, 1, seed, [&] { k_greedy_rounds(s.a); });
    return s.right() ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    return greedy_emu.build(tmp_path_factory.mktemp("greedy"), MAIN)


@pytest.mark.parametrize("missing", [0, 100, 400])
def test_a_full_pool_loses_no_candidate(exe, missing):
    for seed in range(5):
        r = subprocess.run([exe, str(seed), str(missing)], capture_output=True, text=True, timeout=60)
        assert r.returncode == 0, r.stderr
