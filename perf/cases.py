"""The workloads this library is timed on: clustering calls through the public entry points.

Each case is a dict of plain values: the entry point (`entry`), the recipe of the points
(`data`), the dimension, the coordinate type and the number of points (or of sets / jobs).
`prepare` builds on the GPU what a program holds before the call, `run` is one call as a
program makes it, `work` the bytes it cannot do without, `exact` the labels by brute force.
"""
from __future__ import annotations

import math
import random

import torch

import paper_1912_00323_gb300 as hca


def listed():
    return [
        # one small set in double precision, the usual first use of a clustering library: launch
        # and latency bound
        {"name": "small_2d_f64", "entry": "device", "data": "blobs", "d": 2, "f64": True, "n": 10_000},
        # the smallest high-dimensional call: a few thousand feature vectors
        {"name": "small_8d_f32", "entry": "device", "data": "blobs", "d": 8, "f64": False, "n": 3_001},
        # the benchmark workload: a 3-D point cloud of blobs and curved manifolds with noise
        {"name": "cloud_3d_2m", "entry": "device", "data": "manifolds", "d": 3, "f64": False, "n": 2_000_000},
        # the same kind of cloud from a whole survey (more clusters in a larger box), odd size
        {"name": "cloud_3d_16m", "entry": "device", "data": "manifolds", "d": 3, "f64": False, "n": 16_000_003},
        # space-time points in double precision (d = 4, the widest hypercube stencil)
        {"name": "spacetime_4d_f64", "entry": "device", "data": "blobs", "d": 4, "f64": True, "n": 300_001},
        # sensor records in double precision (d = 7, as household power data): FP64 distances
        {"name": "records_7d_f64", "entry": "device", "data": "blobs", "d": 7, "f64": True, "n": 60_007},
        # a mid-sized job of the serving mix in single precision: tensor-core distance tiles
        {"name": "features_9d_f32", "entry": "device", "data": "blobs", "d": 9, "f64": False, "n": 200_003},
        # the high-dimensional benchmark workload: 100 anisotropic clusters in 16 dimensions
        {"name": "aniso_16d_1m", "entry": "device", "data": "anisotropic", "d": 16, "f64": False, "n": 1_000_000},
        # points and labels in host memory: copies, clustering and the read-back in one call
        {"name": "host_2d_f32", "entry": "host", "data": "blobs", "d": 2, "f64": False, "n": 262_147},
        # frames of a sensor clustered one after another by a plan made once for the buffer
        {"name": "plan_3d_frames", "entry": "plan", "data": "manifolds", "d": 3, "f64": False, "n": 150_001},
        # many independent sets of mixed dimension in one call
        {"name": "batched_mixed", "entry": "batched", "data": "blobs", "sets": 128, "n_max": 200_000, "sizes": 1},
        # a burst of jobs of mixed size and dimension through the request server
        {"name": "server_burst", "entry": "server", "data": "blobs", "sets": 32, "n_max": 100_000, "sizes": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["low", "low", "high", "high", "cloud", "host", "plan", "batched", "server"])
    if kind == "low":
        return {"entry": "device", "data": "blobs", "d": rng.randint(1, 4), "f64": rng.random() < 0.5,
                "n": _log_int(rng, 1_000, 1_000_000)}
    if kind == "high":
        if rng.random() < 0.3:
            return {"entry": "device", "data": "blobs", "d": rng.randint(5, 12), "f64": True,
                    "n": _log_int(rng, 1_000, 60_000)}
        return {"entry": "device", "data": "blobs", "d": rng.randint(5, 20), "f64": False,
                "n": _log_int(rng, 1_000, 150_000)}
    if kind == "cloud":
        return {"entry": "device", "data": "manifolds", "d": 3, "f64": rng.random() < 0.25,
                "n": _log_int(rng, 20_000, 8_000_000)}
    if kind == "host":
        return {"entry": "host", "data": "blobs", "d": rng.randint(2, 4), "f64": rng.random() < 0.5,
                "n": _log_int(rng, 2_000, 1_000_000)}
    if kind == "plan":
        d = rng.randint(2, 8)
        return {"entry": "plan", "data": "blobs" if d != 3 else "manifolds", "d": d, "f64": False,
                "n": _log_int(rng, 2_000, 400_000 if d <= 4 else 50_000)}
    if kind == "batched":
        return {"entry": "batched", "data": "blobs", "sets": _log_int(rng, 4, 128),
                "n_max": _log_int(rng, 4_000, 200_000), "sizes": rng.randint(10, 10**6)}
    return {"entry": "server", "data": "blobs", "sets": _log_int(rng, 4, 24), "n_max": _log_int(rng, 4_000, 100_000),
            "sizes": rng.randint(10, 10**6)}


# ---- points -------------------------------------------------------------------------------


def _sets_of(case):
    """(n, d, scale, eps, min_pts) of every set of a batched call or job of a burst: n log-uniform
    from 1,000, the dimensions and scales of the batched and of the serving workload."""
    r = random.Random(case["sizes"])
    dims = (2, 3, 8) if case["entry"] == "batched" else tuple(range(2, 17))
    out = []
    for _ in range(case["sets"]):
        d = r.choice(dims)
        scale = r.uniform(0.5, 3.0) if case["entry"] == "batched" else _blob_scale(d)
        n = _log_int(r, 1_000, case["n_max"])
        out.append((n, d, scale, _blob_eps(n, d, scale), r.randint(4, 16)))
    return out


def _ball(d):
    return math.pi ** (d / 2.0) / math.gamma(d / 2.0 + 1.0)


def _blob_scale(d):
    return 1.5 * math.sqrt(d / 2.0)


def _blob_eps(n, d, scale):
    """The scale of the blobs, or less where the uniform noise alone would put more than one
    point in a ball of that radius (a user's eps tells the clusters from the noise)."""
    return max(1, round(min(scale, 100.0 / (n // 10 * _ball(d)) ** (1.0 / d)) * 4096)) / 4096


def _lattice(x, bits):
    s = float(2 ** bits)
    return torch.round(x * s) / s


def _shuffled(parts, g):
    x = torch.cat(parts)
    return x[torch.randperm(len(x), generator=g, device=x.device)]


def _even(total, parts):
    return [total // parts + (1 if k < total % parts else 0) for k in range(parts)]


def _rand(shape, lo, hi, g):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _randn(shape, g):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _blobs(n, d, scale, g):
    """5 Gaussian blobs (centres U[10, 90]^d) and 10% uniform noise in [0, 100]^d on the 2^-12
    lattice; blob sigma 2 scale / sqrt(d), at most the one that leaves a typical blob point about
    40 neighbours in a ball of that scale."""
    noise = n // 10
    dense = ((n - noise) / 5.0 * _ball(d) / 40.0) ** (1.0 / d)
    sigma = min(2.0 * scale / math.sqrt(d), scale * dense * math.exp(-0.5) / math.sqrt(2.0 * math.pi))
    parts = [_rand(d, 10.0, 90.0, g) + sigma * _randn((m, d), g) for m in _even(n - noise, 5)]
    parts.append(_rand((noise, d), 0.0, 100.0, g))
    return _lattice(_shuffled(parts, g), 12)


def _rotation(d, g):
    q, r = torch.linalg.qr(_randn((d, d), g).cpu())
    return (q * torch.sign(torch.diagonal(r))).cuda()


def _manifolds(n, g):
    """Per 2 million points 40 Gaussian blobs (sigma U[0.5, 3], 80%), 8 noisy arcs (15%) and 5%
    uniform noise in a cube of 1000 per side, the cube and the counts growing with n."""
    scale = max(1.0, n / 2e6)
    box = 1000.0 * scale ** (1.0 / 3.0)
    blobs, arcs = int(round(40 * scale)), int(round(8 * scale))
    n_blob, n_arc = int(round(0.80 * n)), int(round(0.15 * n))
    parts = []
    for m in _even(n_blob, blobs):
        c = _rand(3, 0.05 * box, 0.95 * box, g)
        parts.append(c + _randn((m, 3), g) * _rand(1, 0.5, 3.0, g))
    for m in _even(n_arc, arcs):
        c = _rand(3, 0.1 * box, 0.9 * box, g)
        rot = _rotation(3, g)
        radius, start, span = _rand(1, 20.0, 100.0, g), _rand(1, 0.0, 2 * math.pi, g), _rand(1, 0.5 * math.pi, 2 * math.pi, g)
        th = (start + span * _rand(m, 0.0, 1.0, g))[:, None]
        parts.append(c + radius * (torch.cos(th) * rot[:, 0] + torch.sin(th) * rot[:, 1]) + 0.75 * _randn((m, 3), g))
    parts.append(_rand((n - n_blob - n_arc, 3), 0.0, box, g))
    return _lattice(_shuffled(parts, g), 16)


def _anisotropic(n, d, g):
    """100 Gaussian clusters with rotated diagonal sigmas U[0.2, 1] (90%) and 10% uniform noise
    in [0, 100]^d on the 2^-12 lattice."""
    n_cl = int(round(0.9 * n))
    parts = []
    for m in _even(n_cl, 100):
        parts.append(_rand(d, 10.0, 90.0, g) + (_randn((m, d), g) * _rand(d, 0.2, 1.0, g)) @ _rotation(d, g).T)
    parts.append(_rand((n - n_cl, d), 0.0, 100.0, g))
    return _lattice(_shuffled(parts, g), 12)


def _eps_min_pts(case):
    if case["data"] == "blobs":
        return _blob_eps(case["n"], case["d"], _blob_scale(case["d"])), 5
    return (2.0, 10) if case["data"] == "manifolds" else (4.0, 20)


def _points(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["data"] == "manifolds":
        x = _manifolds(case["n"], g)
    elif case["data"] == "anisotropic":
        x = _anisotropic(case["n"], case["d"], g)
    else:
        x = _blobs(case["n"], case["d"], _blob_scale(case["d"]), g)
    return x.to(torch.float64 if case["f64"] else torch.float32).contiguous()


def _point_sets(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return [_blobs(n, d, scale, g).to(torch.float32).contiguous() for n, d, scale, _, _ in _sets_of(case)]


# ---- what a program holds, and its call ----------------------------------------------------

_server = None


def _the_server():
    """A serving program keeps one server."""
    global _server
    if _server is None:
        _server = hca.Server(device=0, hbm_budget_bytes=32 << 30, workers=4)
    return _server


def prepare(case, seed):
    st = {"entry": case["entry"]}
    if case["entry"] == "batched":
        sets = _sets_of(case)
        st["points"], st["offsets"], st["dims"] = hca.pack_sets(_point_sets(case, seed))
        st["eps"], st["min_pts"] = [s[3] for s in sets], [s[4] for s in sets]
        st["core"] = torch.empty(int(st["offsets"][-1]), dtype=torch.uint8, device="cuda")
        return st
    if case["entry"] == "server":
        st["server"] = _the_server()
        st["jobs"] = [(x.cpu().pin_memory(), e, m) for x, (_, _, _, e, m) in zip(_point_sets(case, seed), _sets_of(case))]
        return st
    x = _points(case, seed)
    st["eps"], st["min_pts"] = _eps_min_pts(case)
    if case["entry"] == "host":
        st["points"] = x.cpu().pin_memory()
        st["labels"] = torch.empty(case["n"], dtype=torch.int32).pin_memory()
        return st
    st["points"] = x
    st["core"] = torch.empty(case["n"], dtype=torch.uint8, device="cuda")
    if case["entry"] == "plan":  # the sensor's range, known before any frame
        lo, hi = -64.0, 1064.0 if case["data"] == "manifolds" else 164.0
        st["plan"] = hca.Plan(x, st["eps"], st["min_pts"], [lo] * case["d"], [hi] * case["d"], core=st["core"])
    return st


def run(st):
    if st["entry"] == "device":
        labels = hca.hca_dbscan_device(st["points"], st["eps"], st["min_pts"], core=st["core"])
        return {"labels": labels, "core": st["core"]}
    if st["entry"] == "host":
        return {"labels": hca.hca_dbscan(st["points"], st["eps"], st["min_pts"], labels=st["labels"])}
    if st["entry"] == "plan":
        st["plan"].launch()
        st["plan"].wait()
        return {"labels": st["plan"].labels, "core": st["core"]}
    if st["entry"] == "batched":
        labels = hca.hca_dbscan_batched(st["points"], st["offsets"], st["eps"], st["min_pts"], dims=st["dims"],
                                        core=st["core"])
        return {"labels": labels, "core": st["core"]}
    tickets = [st["server"].submit(x, e, m) for x, e, m in st["jobs"]]
    return {"labels": [st["server"].wait(t)[0] for t in tickets]}


def work(case):
    """Every coordinate read once, every label (and core flag, where it is asked for) written once."""
    if "sets" in case:
        flag = 1 if case["entry"] == "batched" else 0
        return {"bytes": sum(n * (4 * d + 4 + flag) for n, d, _, _, _ in _sets_of(case)), "flops": 0}
    esz = 8 if case["f64"] else 4
    return {"bytes": case["n"] * (case["d"] * esz + 4 + (case["entry"] != "host")), "flops": 0}


# ---- the definition, by brute force --------------------------------------------------------


def _dbscan(x, eps, min_pts):
    """Labels and core flags of DBSCAN in 64 bits: core points have at least min_pts points
    within eps (themselves included); a cluster's label is its smallest core index; another
    point takes the smallest label among the core points within eps, else -1."""
    x = x.to(torch.float64)
    n, d = x.shape
    step = max(1, (1 << 26) // n)

    def near(i):
        s = torch.zeros((min(step, n - i), n), dtype=torch.float64, device=x.device)
        for k in range(d):
            t = x[i:i + step, k, None] - x[None, :, k]
            s += t * t
        return s <= eps * eps

    adj = torch.cat([near(i) for i in range(0, n, step)])
    core = adj.sum(1) >= min_pts
    none = n
    label = torch.where(core, torch.arange(n, device=x.device), none)
    while True:
        best = torch.cat([torch.where(adj[i:i + step] & core[None, :], label[None, :], none).amin(1)
                          for i in range(0, n, step)])
        new = torch.where(core, torch.minimum(best, label), label)
        new = torch.where(core, new[new.clamp(max=n - 1)], none)
        if torch.equal(new, label):
            break
        label = new
    return torch.where(best == none, -1, best).to(torch.int32), core.to(torch.uint8)


def exact(case, seed):
    if "sets" in case or case["n"] > 12_000:
        return None
    eps, min_pts = _eps_min_pts(case)
    labels, core = _dbscan(_points(case, seed), eps, min_pts)
    return {"labels": labels} if case["entry"] == "host" else {"labels": labels, "core": core}
