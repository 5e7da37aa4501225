"""The waits of the one-pass sorts and scans are bounded.  One that runs out leaves incomplete tables: the call
must end with a status, and nothing after it may read or write by those tables.  A small program
(device/look_back_limit.cu) makes the waits run out with a limit of 256 polls."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_waits_that_run_out(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_00323_gb300 import build
    exe = str(tmp_path / "look_back_limit")
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "device", "look_back_limit.cu"), "-o", exe],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "FAIL" not in r.stdout, r.stdout + r.stderr
