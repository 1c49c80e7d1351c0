"""Calls from a thread with a small stack: results are not staged in arrays on it. On the host, with no GPU (fake_cuda), in a
process of its own."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r"""
import sys, threading
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import numpy as np
import fake_cuda
import paper_1709_03565_gb300 as skis
s = fake_cuda.Sketch(6000)
assert s.sample(1000) == 0
out = []
def run():
    for k in (1, 10, 4096, 4097):
        seeds, cov, est = np.full(k, -1, np.int32), np.full(k, -1, np.int64), np.full(k, -1.0)
        rc = s.fk.skis_greedy_maxcover(s.s, k, seeds.ctypes.data, cov.ctypes.data, est.ctypes.data, None)
        out.append((rc, (seeds == 0).all() and (cov == 0).all() and (est == 0).all()))  # no kernel ran
threading.stack_size(64 << 10)
t = threading.Thread(target=run)
t.start()
t.join()
assert len(out) == 4 and all(rc == 0 and same for rc, same in out), out
s.close()
print("done")
"""


def test_greedy_on_a_64_kib_stack():
    r = subprocess.run([sys.executable, "-c", CODE, ROOT], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "done" in r.stdout, (r.returncode, r.stderr)
