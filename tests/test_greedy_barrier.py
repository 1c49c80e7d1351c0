"""Greedy's kernel when a grid barrier's wait runs out: the block ends without reading by what the barrier did not bring
in (other blocks' candidates, pool entries that were never written). On the host; memory past every array is unreadable."""
import subprocess

import pytest

import greedy_emu

MAIN = r"""
int main(int argc, char** argv) {
    Sketch s(3000, 300, 30, atoi(argv[2]), 2, 1);
    barriers_left = atoi(argv[1]);
    if (argv[3][0] == 's') {  // no room for a pool: segments are scanned
        uint32_t all = 0;
        for (int i = 0; i < kBuckets; ++i) {
            all += s.a.hist[i];
            s.a.hist[i] = 0;
        }
        s.a.hist[kBuckets - 1] = all;
    }
    other_blocks = [&] { s.a.partial[1] = no_cand(); };
    emu::run(kGreedyThreads, 0, 2, 1, [&] { k_greedy_rounds(s.a); });
    return barriers_left == -1 ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    return greedy_emu.build(tmp_path_factory.mktemp("greedy"), MAIN)


# a refill has one grid barrier (its next ones two), a scan of the segments one, the end of a round two
@pytest.mark.parametrize("form", ["pool", "segments"])
@pytest.mark.parametrize("barrier", range(7))
def test_a_block_ends_at_the_barrier_that_ran_out(exe, form, barrier):
    r = subprocess.run([exe, str(barrier), "4", form], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stderr)
