"""The edges of the rules that choose a kernel or a layout, each against the CPU oracle.

Labels and core flags are integers and must be bit-identical, so every tolerance is zero."""
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
    import oracle
    oracle.build()
    import paper_1912_00323_gb300 as pkg
    pkg.load()
    return torch, pkg, oracle


def run(env, X, eps, min_pts, **kw):
    """labels, core flags and stats of one device call"""
    torch, pkg, _ = env
    t = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    core = torch.empty(len(X), dtype=torch.uint8, device="cuda")
    lab, stats = pkg.hca_dbscan_device(t, eps, min_pts, core=core, timing=True, **kw)
    torch.cuda.synchronize()
    return lab.cpu().numpy(), core.cpu().numpy(), stats


def check(got, want):
    bad = np.flatnonzero(got[0] != want[0])
    assert len(bad) == 0, f"{len(bad)} labels differ, first at {bad[:5]}"
    np.testing.assert_array_equal(got[1], want[1])


def clumps(n, extent, seed, per=12, width=2.0):
    """Clumps of `per` points on a 0.25 lattice in the box [0, extent], its corners among them."""
    rng = np.random.default_rng(seed)
    extent = np.asarray(extent, np.float64)
    c = rng.uniform(0, 1, ((n + per - 1) // per, len(extent))) * extent
    X = np.repeat(c, per, axis=0)[:n] + rng.uniform(-width, width, (n, len(extent)))
    X = np.clip(np.round(X * 4) / 4, 0, np.floor(extent * 4) / 4)
    X[0], X[-1] = 0, np.floor(extent * 4) / 4
    return X


@pytest.mark.parametrize("extent", [4.0e4, 2.0e5], ids=["keys32", "keys64"])
@pytest.mark.parametrize("n", [2047, 2048, 2049, 307200, 307201, 614400, 614401, 1228800, 1228801, 13312 * 151 + 5,
                               4000000, 4000001])
def test_sort_tile_sizes(env, n, extent):
    """Sort tiles of 1024 threads x 2, 4, 8 and 13 keys and of 512 x 13, at the ends of each rule and at
    ragged last tiles, with keys of 32 and of 64 bits; so too the one-pass scans over the cells,
    and early launches, which end at 2^21 points."""
    X = clumps(n, (extent, extent), seed=n, per=40)
    want = env[2].grid(X, 1.25, 5)
    got = run(env, X.astype(np.float32), 1.25, 5)
    check(got, want)
    assert (got[2]["key_bits"] > 32) == (extent > 1e5)


@pytest.mark.parametrize("n", [1, 14, 15, 16, 17, 31, 33, 1000])
@pytest.mark.parametrize("offset", [0, 1, 15])
def test_core_flags_at_any_alignment(env, n, offset):
    """Core flags are set in 16-byte stores first: unaligned starts, ragged ends, bytes around them."""
    torch, pkg, oracle = env
    X = clumps(n, (40.0, 40.0), seed=n)
    want = oracle.grid(X, 1.25, 5)
    out = torch.full((n + 48,), 7, dtype=torch.uint8, device="cuda")
    lab = pkg.hca_dbscan_device(torch.from_numpy(X).cuda(), 1.25, 5, core=out[offset:offset + n])
    torch.cuda.synchronize()
    check((lab.cpu().numpy(), out[offset:offset + n].cpu().numpy()), want)
    rest = torch.cat([out[:offset], out[offset + n:]])
    assert bool((rest == 7).all())
