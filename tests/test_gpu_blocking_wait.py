"""A program that asks its device for blocking waits gets them: the calls do not poll.  The flag belongs to the
process's context, so the check runs in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes, sys, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(0, int(sys.argv[1])) == 0
sys.path.insert(0, sys.argv[2])
import torch
import paper_1912_00323_gb300 as pkg
x = torch.rand((1_000_000, 3), device="cuda") * 400
for _ in range(5):
    lab = pkg.hca_dbscan_device(x, 2.0, 5, graph_cache=False)
w, t = time.perf_counter(), time.thread_time()
for _ in range(200):
    pkg.hca_dbscan_device(x, 2.0, 5, labels=lab, graph_cache=False)
print((time.thread_time() - t) / (time.perf_counter() - w))
"""


def busy(flags):
    """Share of the wall time that the calling thread runs."""
    r = subprocess.run([sys.executable, "-c", CHILD, str(flags), ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    return float(r.stdout)


def test_blocking_waits():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spin, block = busy(1), busy(4)  # CU_CTX_SCHED_SPIN, CU_CTX_SCHED_BLOCKING_SYNC
    assert block < 0.25 and spin > 2 * block, (spin, block)  # (with the polls 0.39, without 0.08; spinning 1)
