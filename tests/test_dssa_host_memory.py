"""skis_dssa_maxinf without the host memory for k seeds' results returns SKIS_ENOMEM: no exception leaves the library. On the
host, with no GPU (fake_cuda), in a process of its own whose address space is limited."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r"""
import sys, resource, ctypes
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import numpy as np
import fake_cuda
import paper_1709_03565_gb300 as skis
n = 1 << 28
s = fake_cuda.Sketch(n)
seeds = np.empty(16, np.int32)  # never written: the call fails first
res = skis._binding.skis_dssa_result()
size = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (size + (1 << 30), resource.RLIM_INFINITY))  # 2 GiB are asked for at a time
rc = s.fk.skis_dssa_maxinf(s.g, 1, 2, n, 0.1, 0.1, 0, 100, 1000, seeds.ctypes.data, ctypes.byref(res), None)
assert rc == skis.SKIS_ENOMEM, rc
assert s.fk.skis_last_error().startswith(b"skis_dssa_maxinf")
s.close()
print("done")
"""


def test_no_exception_leaves_the_library():
    r = subprocess.run([sys.executable, "-c", CODE, ROOT], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "done" in r.stdout, (r.returncode, r.stderr)
