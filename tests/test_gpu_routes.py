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


@pytest.mark.parametrize("d,extent", [(1, 9.0e5), (3, 40.0), (3, 3000.0), (4, 30.0), (4, 500.0)])
@pytest.mark.parametrize("n", [2047, 2049, 40000])
def test_pencil_table_and_hash(env, d, extent, n):
    """Neighbour pencils through the direct table (few pencil keys for the points) and through the hash
    table (the wide boxes of 3-D and 4-D), at the edges of the 2,048-point tiles of the cells."""
    X = clumps(n, (extent,) * d, seed=n + d, per=20)
    want = env[2].grid(X, 1.75, 6)
    check(run(env, X, 1.75, 6), want)


@pytest.mark.parametrize("n", [499999, 500000, 500001])
def test_representative_windows(env, n):
    """Windows of 32 points below 500,000, of 64 from there; cells across window ends."""
    X = clumps(n, (220.0, 220.0, 220.0), seed=n, per=50, width=2.0)
    want = env[2].grid(X, 1.25, 6)
    check(run(env, X.astype(np.float32), 1.25, 6), want)


@pytest.mark.parametrize("n", [2 ** 20, 2 ** 20 + 1])
@pytest.mark.parametrize("d", [2, 6])
def test_batched_early_launches(env, n, d):
    """Batched calls put their kernels in place early up to 2^20 points: sets of very unequal size."""
    torch, pkg, oracle = env
    sizes = [n - 1203, 1, 2, 200, 1000]
    X = [clumps(m, (300.0,) * min(d, 3) + (6.0,) * (d - 3), seed=m + d, per=60, width=0.4) for m in sizes]
    flat, off, dims = pkg.pack_sets([x.astype(np.float32) for x in X])
    lab = pkg.hca_dbscan_batched(flat, off, [1.25] * 5, [5, 1, 2, 7, 5], dims=dims).cpu().numpy()
    for s, mp in enumerate([5, 1, 2, 7, 5]):
        np.testing.assert_array_equal(lab[off[s]:off[s + 1]], oracle.grid(X[s], 1.25, mp)[0], err_msg=f"set {s}")


def lists(n, d, seed):
    """Lattice clumps of 1 to 150 points and single points between them: many pairs at exactly eps, cells with
    and without core points, clusters that only border points touch."""
    rng = np.random.default_rng(seed)
    X, left = [], n
    while left > 0:
        m = min(left, int(rng.integers(1, 150)))
        X.append(rng.uniform(0, 12, d) + rng.uniform(-1, 1, (m, d)) * rng.uniform(0.2, 1.5))
        left -= m
    return np.round(np.concatenate(X) * 4) / 4


@pytest.mark.parametrize("min_pts", [1, 2, 9, 10, 20, 21, 22, 60, 400])
@pytest.mark.parametrize("d", [5, 9, 16])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_neighbour_lists(env, d, min_pts, dtype):
    """MINPTS up to 21 is labelled from complete neighbour lists (20 entries), above by comparison; every point
    core, hardly any, and counts that start again on long rows; with the tensor cores and without."""
    X = lists(5000, d, seed=d)
    eps = 0.25 * round(4 * (0.45 * d ** 0.5 + 0.3))
    want = env[2].grid(X, eps, min_pts)
    check(run(env, X.astype(dtype), eps, min_pts), want)
    if dtype == np.float32:
        check(run(env, X.astype(dtype), eps, min_pts, tensor_cores=False), want)


@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (4096.0, 1.0), (2.0 ** 30, 1.0), (0.0, 2.0 ** -60), (0.0, 2.0 ** 70)])
@pytest.mark.parametrize("d", [5, 8])
def test_float_filter_of_doubles(env, d, shift, scale):
    """A float copy relative to the minimum decides most pairs of double input: ties on a lattice, large offsets
    (exact in double), scales where eps^2 leaves the filter's range, a far point that makes it coarse; the same
    labels with every pair in double."""
    for far in (0.0, 2.0 ** 20):
        X = lists(3000, d, seed=3 * d)
        if far:
            X[1234, 0] = far
        eps = 0.25 * round(2 * d ** 0.5 + 1) * scale
        X = (X + shift) * scale
        want = env[2].grid(X, eps, 7)
        check(run(env, X, eps, 7), want)
        check(run(env, X, eps, 7, fp64_only=True), want)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("min_pts", [5, 3000])
def test_long_streams_spill(env, dtype, min_pts):
    """Streams of far more than 1,024 candidates on the CUDA cores, whose rest is counted, labelled and joined in
    windows of a second launch: one dense ball, a thin shell of border points and noise around it."""
    rng = np.random.default_rng(5)
    v = rng.normal(size=(9000, 6))
    r = np.concatenate([rng.uniform(0, 1.0, 8000), rng.uniform(1.8, 2.6, 1000)])
    X = np.round(v / np.linalg.norm(v, axis=1, keepdims=True) * r[:, None] * 64) / 64
    want = env[2].grid(X, 1.5, min_pts)
    check(run(env, X.astype(dtype), 1.5, min_pts, tensor_cores=False), want)


def test_batched_doubles_of_any_offset(env):
    """Batched double sets share a call whose float copies are relative to each set's own minimum."""
    torch, pkg, oracle = env
    X = [lists(m, 7, seed=m) + o for m, o in ((3000, 0.0), (1, 5.0), (2047, 1.0e9), (500, -2.0 ** 33), (4097, 3.0))]
    off = np.concatenate([[0], np.cumsum([len(x) for x in X])])
    eps, mp = [1.25, 1.0, 1.5, 1.75, 1.5], [6, 1, 4, 22, 30]
    lab = pkg.hca_dbscan_batched(torch.from_numpy(np.concatenate(X)).cuda(), off, eps, mp).cpu().numpy()
    for s in range(5):
        np.testing.assert_array_equal(lab[off[s]:off[s + 1]], oracle.grid(X[s], eps[s], mp[s])[0], err_msg=f"set {s}")


@pytest.mark.parametrize("sets", [1, 16, 17, 256, 257])
@pytest.mark.parametrize("d", [3, 6])
def test_extents_by_mail_and_by_copy(env, sets, d):
    """The extents of up to 2,048 words (256 sets of d <= 4, 16 above) come through the pinned mailbox, of more by
    a copy."""
    torch, pkg, oracle = env
    X = [clumps(30 + s, (20.0 + s,) * d, seed=s) + s for s in range(sets)]
    off = np.concatenate([[0], np.cumsum([len(x) for x in X])])
    lab = pkg.hca_dbscan_batched(torch.from_numpy(np.concatenate(X)).cuda(), off, [1.5] * sets, [4] * sets).cpu().numpy()
    for s in range(sets):
        np.testing.assert_array_equal(lab[off[s]:off[s + 1]], oracle.grid(X[s], 1.5, 4)[0], err_msg=f"set {s}")
