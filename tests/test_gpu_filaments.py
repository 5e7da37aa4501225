"""Points along a line: one cluster whose first links chain up over all of its cells (d <= 4) or
points (d >= 5), flattened by jumps of all nodes together."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_00323_gb300 import build
    build.build()
    import paper_1912_00323_gb300 as pkg
    pkg.load()
    return torch, pkg


def line(torch, n, d, step):
    """n points `step` apart in every coordinate, shuffled, a gap of 8 in the middle."""
    t = np.arange(n) * step
    t[n // 2:] += 8.0
    t = t[np.random.default_rng(n + d).permutation(n)]
    want = np.where(t < (n // 2) * step, np.argmin(np.where(t < (n // 2) * step, 0, 1)),
                    np.argmin(np.where(t < (n // 2) * step, 1, 0)))
    return torch.from_numpy(np.repeat(t[:, None], d, axis=1)).cuda(), want


@pytest.mark.parametrize("n", [3, 130, 20_000, 700_000])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 9])
def test_two_lines(env, n, d):
    """Every point has a neighbour within eps = 1 on its line: two clusters, all points core."""
    torch, pkg = env
    n = min(n, 60_000) if d == 4 else n  # (16 bits of every coordinate would not fit the keys)
    X, want = line(torch, n, d, 0.25)
    if n == 3:  # a single point and a pair
        want = np.where(want == np.bincount(want).argmax(), want, -1)
    np.testing.assert_array_equal(pkg.hca_dbscan_device(X, 1.0, 2).cpu().numpy(), want)


def test_time_along_a_line(env):
    """A cell and a half a point, each core by its two neighbours: the merge stage of the call stays in
    the order of its count stage (about 1.3 times; walking the links one by one 3.5 times)."""
    torch, pkg = env
    X, want = line(torch, 1_000_000, 1, 0.75)
    best = {}
    for _ in range(8):
        lab, st = pkg.hca_dbscan_device(X, 1.0, 3, timing=True)
        for k, v in st["stage_ms"].items():
            best[k] = min(v, best.get(k, v))
    np.testing.assert_array_equal(np.unique(lab.cpu().numpy(), return_inverse=True)[1],
                                  np.unique(want, return_inverse=True)[1])  # (the ends are border points)
    assert best["merge"] < 2.2 * best["core"], best
