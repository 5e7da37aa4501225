"""The float filter of double input (d >= 5) on points of no lattice, whose float copies round: stars of points
whose distances to their centre are eps (1 +- 1e-9 .. 1e-4), far apart from each other.  A float sum of
squares below lo32 says within, above hi32 outside; the thresholds leave room for the rounding of the copies,
and what lies between them is decided in double.

On the CPU the filter is emulated: no pair is decided wrongly, and with the room taken out some are, so
the points would show it.  On the GPU labels and core flags are compared with the oracle's."""
import math

import numpy as np
import pytest

CASES = [(5, 0.0, 30.0), (7, 1.0e9, 30.0), (8, -3.0, 200.0), (16, 5.0e5, 60.0), (33, 0.1, 40.0), (64, 7.0, 30.0)]
EPS = 0.7371


def stars(d, offset, box, seed=11):
    """Centres in [0, box]^d + offset and twelve points around each."""
    rng = np.random.default_rng(seed + d)
    c = rng.uniform(0, box, (250, d))
    parts = [c]
    for k in range(12):
        v = rng.normal(size=c.shape)
        v /= np.linalg.norm(v, axis=1, keepdims=True)
        r = EPS * (1 + rng.choice([-1, 1], 250) * 10.0 ** rng.uniform(-9, -4, 250))
        parts.append(c + v * r[:, None])
    X = np.concatenate(parts) + offset
    return X[rng.permutation(len(X))]


def f32_up(x):
    f = np.float32(x)
    return f if float(f) >= x else np.nextafter(f, np.float32(np.inf))


def f32_down(x):
    f = np.float32(x)
    return f if float(f) <= x else np.nextafter(f, np.float32(0))


def thresholds(X, room):
    ext = np.linalg.norm(X.max(0) - X.min(0))
    off = 2.0 ** -23 * (1 + 2.0 ** -20) * ext if room else 0.0
    assert off <= 0.25 * EPS
    g = 2.0 ** -16 if room else 0.0
    return f32_down((EPS - off) ** 2 * (1 - g)), f32_up((EPS + off) ** 2 * (1 + g))


def float_sums(X, i, j):
    """The device's sum: float copies relative to the minimum, even and odd dimensions by fused
    multiply-adds (the product is exact in double), then one addition."""
    F = (X - X.min(0)).astype(np.float32)
    s = [np.zeros(len(i), np.float32), np.zeros(len(i), np.float32)]
    for k in range(X.shape[1]):
        t = (F[i, k] - F[j, k]).astype(np.float64)
        s[k % 2] = (s[k % 2].astype(np.float64) + t * t).astype(np.float32)
    return s[0] + s[1]


def exact(X, i, j):
    s = np.zeros(len(i))
    for k in range(X.shape[1]):
        t = X[i, k] - X[j, k]
        s = s + t * t
    return s <= EPS * EPS


@pytest.mark.parametrize("d,offset,box", CASES)
def test_filter_decides_no_pair_wrongly(d, offset, box):
    X = stars(d, offset, box)
    from scipy.spatial import cKDTree
    i, j = cKDTree(X).query_pairs(EPS * 1.01, output_type="ndarray").T
    assert len(i) >= 2900
    s, inside = float_sums(X, i, j), exact(X, i, j)
    lo, hi = thresholds(X, True)
    assert not np.any((s < lo) & ~inside) and not np.any((s > hi) & inside)
    lo, hi = thresholds(X, False)
    assert np.any((s < lo) & ~inside) and np.any((s > hi) & inside)


@pytest.mark.gpu
@pytest.mark.parametrize("min_pts", [2, 6, 7, 30])
@pytest.mark.parametrize("d,offset,box", CASES)
def test_labels_off_the_lattice(d, offset, box, min_pts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_00323_gb300 import build
    build.build()
    import oracle
    oracle.build()
    import paper_1912_00323_gb300 as pkg
    X = stars(d, offset, box)
    want, want_core = oracle.grid(X, EPS, min_pts)
    core = torch.empty(len(X), dtype=torch.uint8, device="cuda")
    for fp64_only in (False, True):
        lab = pkg.hca_dbscan_device(torch.from_numpy(X).cuda(), EPS, min_pts, core=core, fp64_only=fp64_only)
        np.testing.assert_array_equal(lab.cpu().numpy(), want)
        np.testing.assert_array_equal(core.cpu().numpy(), want_core)
