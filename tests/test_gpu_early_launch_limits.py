"""Calls on either side of the sizes up to which their kernels are put in place early (2^21 points, 2^20 on the
coarse grid), against the CPU oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def clumps(n, extent, seed, per, width):
    rng = np.random.default_rng(seed)
    extent = np.asarray(extent, np.float64)
    c = rng.uniform(0, 1, ((n + per - 1) // per, len(extent))) * extent
    X = np.repeat(c, per, axis=0)[:n] + rng.uniform(-width, width, (n, len(extent)))
    return np.clip(np.round(X * 4) / 4, 0, np.floor(extent * 4) / 4).astype(np.float32)


@pytest.mark.parametrize("n,extent,per,width", [
    (2 ** 21, (2.0e4, 2.0e4), 40, 2.0), (2 ** 21 + 1, (2.0e4, 2.0e4), 40, 2.0),
    (2 ** 20, (300.0, 300.0, 300.0, 6.0, 6.0, 6.0), 60, 0.4), (2 ** 20 + 1, (300.0, 300.0, 300.0, 6.0, 6.0, 6.0), 60, 0.4)])
def test_single_sets(n, extent, per, width):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_00323_gb300 import build
    build.build()
    import oracle
    oracle.build()
    import paper_1912_00323_gb300 as pkg
    X = clumps(n, extent, n, per, width)
    want, want_core = oracle.grid(X.astype(np.float64), 1.25, 5)
    core = torch.empty(n, dtype=torch.uint8, device="cuda")
    lab = pkg.hca_dbscan_device(torch.from_numpy(X).cuda(), 1.25, 5, core=core, graph_cache=False)
    np.testing.assert_array_equal(lab.cpu().numpy(), want)
    np.testing.assert_array_equal(core.cpu().numpy(), want_core)
