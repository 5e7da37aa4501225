"""Coarse-grid calls and plans without memory for whole neighbour lists run with short ones in the space of the
pencil table: same labels, and a workspace no larger than it was without lists."""
import glob
import os
import subprocess

import pytest

from paper_1912_00323_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _objects():
    build.build()
    objs = glob.glob(os.path.join(build.BUILD, "*.o"))
    if len(objs) < len(build.SOURCES):
        build.build(force=True)
        objs = glob.glob(os.path.join(build.BUILD, "*.o"))
    return sorted(objs)


@pytest.mark.gpu
def test_no_memory_for_lists(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = str(tmp_path / "scratch_limit")
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC,
                    os.path.join(ROOT, "tests", "device", "scratch_limit.cu"), *_objects(),
                    "-Xlinker", "--wrap=_ZN3hca10pool_allocEPPvmP11CUstream_st", "-o", exe],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "FAIL" not in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("d,dtype,bytes_per_point", [(8, "float32", 360), (16, "float32", 456), (7, "float64", 416)])
def test_bound_per_point(d, dtype, bytes_per_point):
    """The lists share the table's space: 76 bytes a point became 28 to 52."""
    import paper_1912_00323_gb300 as pkg
    for n in (200_003, 1_000_000, 2 ** 20, 2 ** 20 + 1):
        assert pkg.hca_workspace_bytes(n, d, dtype) < bytes_per_point * n


@pytest.mark.gpu
@pytest.mark.parametrize("budget", [1, 64 << 20, 8 << 30])
def test_server_budgets(budget):
    """Jobs with whole lists, with short ones (a budget with no room for more, jobs larger than it alone) and
    mixed: the labels of a call of their own."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np
    import paper_1912_00323_gb300 as pkg
    rng = np.random.default_rng(3)
    jobs = []
    for k in range(40):
        d, n = [5, 9, 16, 3][k % 4], int(rng.integers(500, 30_000))
        c = rng.uniform(0, 30, (n // 60 + 1, d)).repeat(60, axis=0)[:n]
        X = np.round((c + rng.normal(size=(n, d)) * 0.5) * 64) / 64
        jobs.append((X.astype(np.float32 if k % 3 else np.float64), 0.9 * d ** 0.5, [2, 6, 12, 21, 40][k % 5]))
    with pkg.Server(hbm_budget_bytes=budget, workers=3) as sv:
        tickets = [sv.submit(*j) for j in jobs]
        got = [sv.wait(t)[0] for t in tickets]
    for (X, eps, mp), lab in zip(jobs, got):
        np.testing.assert_array_equal(lab, pkg.hca_dbscan(X, eps, mp))
