"""Sampling on a GPU whose memory is mostly taken: the default scratch and the first arena's 2 GiB have no room, the samples
are the oracle's all the same. In a process of its own, which holds the memory."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r"""
import sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import numpy as np, torch
import oracle, synth
import paper_1709_03565_gb300 as skis
from test_gpu_parity import assert_samples_equal
n, T = 200_000, 4_000_000
src, dst = synth.er(n, 1_000_000, 3)
warm = skis.skis_load_graph(1000, src[:2000] % 999, src[:2000] % 999 + 1, weight_model=skis.SKIS_W_WC)
s = skis.skis_sketch_create(warm, 1)  # the library's kernels are loaded while there is room
skis.skis_sample(s, 1000)
s.close()
warm.close()
g = skis.skis_load_graph(n, src, dst, weight_model=skis.SKIS_W_TRI, weight_seed=5)
torch.cuda.synchronize()
hold = torch.empty(torch.cuda.mem_get_info()[0] - (3 << 29), dtype=torch.uint8, device="cuda")
s = skis.skis_sketch_create(g, 77)
skis.skis_sample(s, T)
st = skis.skis_sketch_stats(s)
assert st["T"] == T and st["arena_capacity"] < 1 << 28, st
o = oracle.OracleGraph(n, src, dst, model=oracle.W_TRI, weight_seed=5)
ids = np.arange(T - 3000, T, dtype=np.uint64)
assert_samples_equal(skis.skis_sketch_export(s, T - 3000, 3000), o.sample_ids(77, ids))
del hold
s.close()
g.close()
print("done")
"""


def test_samples_with_little_memory_left():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.empty_cache()
    r = subprocess.run([sys.executable, "-c", CODE, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stderr[-2000:]
