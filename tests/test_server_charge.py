"""Admission of the request server: a job is charged what its call cannot do without, not the neighbour lists
that it runs faster with.  The charge per point must not exceed the one from before there were lists (point and
label bytes, 16 and 1 KB for the shared call, and the workspace per point listed here); the lists come on top
only where the budget has room for them (host code only, no GPU)."""
import glob
import os
import shutil
import subprocess

import pytest

from paper_1912_00323_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# (n, d, dtype): workspace per point without lists
WITHOUT = {(200_003, 8, 0): 313.9, (1_000_000, 8, 0): 307.4, (2 ** 20 + 1, 8, 0): 330.3, (200_003, 16, 0): 409.9,
           (1_000_000, 16, 0): 403.4, (200_003, 7, 1): 369.8, (2 ** 20, 7, 1): 362.3, (1_000_000, 33, 0): 979.4}


def test_charge(tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("nvcc not available")
    build.build()
    objs = [o for o in glob.glob(os.path.join(build.BUILD, "*.o")) if not o.endswith("server.o")]
    if len(objs) < len(build.SOURCES) - 1:
        build.build(force=True)
        objs = [o for o in glob.glob(os.path.join(build.BUILD, "*.o")) if not o.endswith("server.o")]
    exe = str(tmp_path / "server_charge")
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "host", "server_charge.cu"), *sorted(objs), "-o", exe],
                   check=True, capture_output=True, text=True)
    asked = [(n, d, t, mp) for n, d, t in WITHOUT for mp in (2, 5, 9, 20, 1000)]
    out = subprocess.run([exe], input="".join("%d %d %d %d\n" % a for a in asked), check=True, capture_output=True,
                         text=True).stdout.split("\n")
    for (n, d, t, mp), line in zip(asked, out):
        charge, lists = map(int, line.split())
        assert charge <= n * (d * (4 if t == 0 else 8) + 4 + 16 + WITHOUT[n, d, t]) + 1024, (n, d, t, mp)
        assert 0 <= lists <= 56 * n
        assert lists > 0 if mp >= 20 else True
