"""The clustering calls that this library is measured by.

A case is one call of a public entry point (``dbscan_run``, ``dbscan_run_multi``,
``dbscan_run_batch``, ``dbscan_run_host``) on synthetic points of one of the
workload families (``workloads/generators.py`` describes them; they are drawn
here on the GPU, from a seed):

* ``blobs``: eight Gaussian blobs and 10% noise in the unit cube (small
  clouds, the instances of a batch, the dense jobs of a server);
* ``roads``: GPS-trace-like points along polylines in the unit square;
* ``halos``: NFW halos with a power-law size distribution and a 30% uniform
  background (cosmology particles), eps 0.2 times the mean spacing;
* ``dims``: blobs and background in 4 to 8 dimensions.

Results are labels and core flags of every point: whole numbers, so there is
no 64-bit value to compare them with.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2103_05162_gb300 as gb

DEV = "cuda"


def listed():
    return [
        # The smallest cloud of a batch or of a stream of frames, one call each: launches and latency.
        {"name": "blobs3_1000", "call": "run", "family": "blobs", "dim": 3, "n": 1000, "min_pts": 5,
         "eps": 0.03, "algo": "densebox", "mode": "dbscan"},
        # The small configuration: 16,384 points in 3D.
        {"name": "blobs3_16384", "call": "run", "family": "blobs", "dim": 3, "n": 16384, "min_pts": 5,
         "eps": 0.03, "algo": "densebox", "mode": "dbscan"},
        # A median batch instance in 2D, odd size, on the plain tree, border points dropped.
        {"name": "blobs2_20011_fd_star", "call": "run", "family": "blobs", "dim": 2, "n": 20011, "min_pts": 10,
         "eps": 0.01, "algo": "fdbscan", "mode": "dbscan*"},
        # A mid-sized serving job of cosmology particles.
        {"name": "halos_262144", "call": "run", "family": "halos", "dim": 3, "n": 262144, "min_pts": 10,
         "eps": 0.0, "algo": "densebox", "mode": "dbscan"},
        # A mid-sized set of GPS traces.
        {"name": "roads_524287_fd", "call": "run", "family": "roads", "dim": 2, "n": 524287, "min_pts": 10,
         "eps": 0.0, "algo": "fdbscan", "mode": "dbscan"},
        # Higher-dimensional data: 5D blobs and background.
        {"name": "dims5_400000", "call": "run", "family": "dims", "dim": 5, "n": 400000, "min_pts": 10,
         "eps": 0.03, "algo": "densebox", "mode": "dbscan"},
        # A parameter sweep: four minPts over one index.
        {"name": "sweep_halos_1048576", "call": "multi", "family": "halos", "dim": 3, "n": 1048576,
         "min_pts": "2,5,10,20", "eps": 0.0, "algo": "densebox", "mode": "dbscan"},
        # Host arrays in, host labels out, the library choosing the algorithm; dense data.
        {"name": "host_blobs3_1000003_auto", "call": "host", "family": "blobs", "dim": 3, "n": 1000003,
         "min_pts": 5, "eps": 0.03, "algo": "auto", "mode": "dbscan"},
        # Many small problems in one fused call: lognormal sizes, 2D and 3D mixed.
        {"name": "batch_512", "call": "batch", "family": "blobs", "count": 512, "sizes": 4, "algo": "densebox",
         "mode": "dbscan"},
        # The 2D configuration: 4M points of GPS traces.
        {"name": "roads_4194304_fd", "call": "run", "family": "roads", "dim": 2, "n": 4194304, "min_pts": 10,
         "eps": 0.0, "algo": "fdbscan", "mode": "dbscan"},
        # Friends-of-friends halo finding (minPts 2, no preprocessing) at the largest serving size, odd.
        {"name": "halos_8000001_fof_fd", "call": "run", "family": "halos", "dim": 3, "n": 8000001, "min_pts": 2,
         "eps": 0.0, "algo": "fdbscan", "mode": "dbscan"},
        # The benchmark: 16M cosmology particles.
        {"name": "halos_16777216", "call": "run", "family": "halos", "dim": 3, "n": 16777216, "min_pts": 10,
         "eps": 0.0, "algo": "densebox", "mode": "dbscan"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["run"] * 7 + ["multi", "host", "batch"])
    mode = rng.choice(["dbscan", "dbscan", "dbscan*"])
    if call == "batch":
        return {"call": "batch", "family": "blobs", "count": _log_int(rng, 8, 512), "sizes": rng.randrange(1 << 20),
                "algo": "densebox", "mode": mode}
    family = rng.choice(["blobs", "roads", "halos", "halos", "dims"])
    algo = rng.choice(["fdbscan", "densebox", "densebox", "auto"])
    most = 16777216 if call == "run" else 2097152
    if family == "blobs":
        dim = rng.choice([2, 3])
        # (without dense cells the neighbourhoods of a blob grow with n: the plain tree takes the small clouds)
        n = _log_int(rng, 1000, 100000 if algo == "fdbscan" else min(most, 4000000))
        eps = round(rng.uniform(0.01, 0.05), 4) if n <= 500000 else 0.03
    elif family == "roads":
        dim, n, eps = 2, _log_int(rng, 10000, min(most, 8000000)), 0.0
    elif family == "halos":
        dim, n, eps = 3, _log_int(rng, 10000, most), 0.0
    else:
        dim = rng.choice([4, 5, 6, 7, 8])
        n = _log_int(rng, 2000, 400000 if dim <= 5 else 150000)
        eps = round(0.0134 * math.sqrt(dim), 4)
    min_pts = "2,5,10,20" if call == "multi" else rng.choice([2, 5, 10, 20])
    return {"call": call, "family": family, "dim": dim, "n": n, "min_pts": min_pts, "eps": eps, "algo": algo,
            "mode": mode}


# ---------------------------------------------------------------- the points

def _blobs(n, d, g, n_blobs=8, sigma=0.02, blob_frac=0.9):
    centres = torch.rand(n_blobs, d, device=DEV, generator=g)
    which = torch.randint(0, n_blobs, (n,), device=DEV, generator=g)
    pts = centres[which] + sigma * torch.randn(n, d, device=DEV, generator=g)
    noise = torch.rand(n, d, device=DEV, generator=g)
    return torch.where(torch.rand(n, 1, device=DEV, generator=g) < blob_frac, pts, noise)


def _roads(n, g, n_roads=2000, n_segments=10, jitter=1e-4, road_frac=0.95):
    start = 0.05 + 0.9 * torch.rand(n_roads, 1, 2, device=DEV, generator=g)
    heading = 2.0 * math.pi * torch.rand(n_roads, n_segments, device=DEV, generator=g)
    length = 0.002 + 0.006 * torch.rand(n_roads, n_segments, device=DEV, generator=g)
    steps = torch.stack([heading.cos() * length, heading.sin() * length], dim=-1)
    verts = torch.cat([start, start + steps.cumsum(1)], dim=1).clamp(0.0, 1.0)
    a, b = verts[:, :-1].reshape(-1, 2), verts[:, 1:].reshape(-1, 2)
    cum = (b - a).norm(dim=1).double().cumsum(0)
    u = torch.rand(n, device=DEV, generator=g, dtype=torch.float64) * cum[-1]
    seg = torch.searchsorted(cum, u, right=True).clamp_(max=a.shape[0] - 1)
    t = torch.rand(n, 1, device=DEV, generator=g)
    on = a[seg] + t * (b[seg] - a[seg]) + jitter * torch.randn(n, 2, device=DEV, generator=g)
    noise = torch.rand(n, 2, device=DEV, generator=g)
    return torch.where(torch.rand(n, 1, device=DEV, generator=g) < road_frac, on, noise)


def _halos(n, g, r_s=0.002, conc=10.0, halo_frac=0.7):
    n_halos = max(10, round(50000 * n / 2**24))
    u = torch.rand(n_halos, device=DEV, generator=g, dtype=torch.float64)
    cum = (1.0 / (0.1 - u * (0.1 - 1e-5))).cumsum(0)  # sizes from p(s) ~ s^-2 on [10, 1e5]
    u = torch.rand(n, device=DEV, generator=g, dtype=torch.float64) * cum[-1]
    halo = torch.searchsorted(cum, u, right=True).clamp_(max=n_halos - 1)
    centres = 0.02 + 0.96 * torch.rand(n_halos, 3, device=DEV, generator=g)
    # radii by the inverse of the enclosed NFW mass, from a table
    x = torch.linspace(0.0, 1.0, 8193, device=DEV, dtype=torch.float64).square() * conc
    mass = torch.log1p(x) - x / (1.0 + x)
    mass = mass / mass[-1]
    u = torch.rand(n, device=DEV, generator=g, dtype=torch.float64)
    k = torch.searchsorted(mass, u, right=True).clamp_(1, mass.numel() - 1)
    w = (u - mass[k - 1]) / (mass[k] - mass[k - 1])
    r = (r_s * (x[k - 1] + w * (x[k] - x[k - 1]))).float()
    v = torch.randn(n, 3, device=DEV, generator=g)
    v = v / v.norm(dim=1, keepdim=True).clamp_(min=1e-20)
    bg = torch.rand(n, 3, device=DEV, generator=g)
    return torch.where(torch.rand(n, 1, device=DEV, generator=g) < halo_frac, centres[halo] + r[:, None] * v, bg)


def _points(family, n, dim, g):
    if family == "roads":
        return _roads(n, g)
    if family == "halos":
        return _halos(n, g)
    if family == "dims":
        return _blobs(n, dim, g, n_blobs=40, blob_frac=0.75)
    return _blobs(n, dim, g)


def _eps(case):
    """0: the neighbourhood of the family, which shrinks as the points get denser."""
    if case["eps"]:
        return float(np.float32(case["eps"]))
    if case["family"] == "roads":
        return float(np.float32(2e-4 * (4194304 / case["n"]) ** 0.5))
    return float(np.float32(0.2 * case["n"] ** (-1.0 / 3.0)))


def _min_pts(case):
    return [int(v) for v in str(case["min_pts"]).split(",")]


def _instances(case):
    """Sizes, dimensions, eps and minPts of a batch (the case's shape; the points come from the seed)."""
    r, count = np.random.Generator(np.random.PCG64(case["sizes"])), case["count"]
    sizes = np.clip(r.lognormal(math.log(20000.0), 1.2, size=count), 1000, 500000).round().astype(np.int64)
    return (sizes, r.choice([2, 3], size=count).astype(np.int32),
            r.uniform(0.01, 0.05, size=count).astype(np.float32), r.choice([2, 5, 10], size=count).astype(np.int32))


# ------------------------------------------------------------------ the calls

def prepare(case, seed):
    # Block size and cell factor as documented for untuned calls, so that two processes sort the points into the
    # same tiles: where a border point has a choice of clusters, the tiles decide which one it joins.
    gb.set_tuning(128, 1.0)
    g = torch.Generator(device=DEV).manual_seed(seed)
    if case["call"] == "batch":
        sizes, dims, eps, min_pts = _instances(case)
        parts = [_blobs(int(n), int(d), g).reshape(-1) for n, d in zip(sizes, dims)]
        return {"case": case, "points": torch.cat(parts), "offsets": np.concatenate([[0], np.cumsum(sizes)]),
                "dims": dims, "eps": eps, "min_pts": min_pts,
                "core": torch.empty(int(sizes.sum()), dtype=torch.uint8, device=DEV)}
    points = _points(case["family"], case["n"], case["dim"], g).contiguous()
    state = {"case": case, "points": points, "eps": _eps(case), "min_pts": _min_pts(case)}
    if case["call"] == "host":
        state["points"] = points.cpu().pin_memory().numpy()
        state["labels"] = torch.empty(case["n"], dtype=torch.int32).pin_memory().numpy()
        state["core"] = torch.empty(case["n"], dtype=torch.uint8).pin_memory().numpy()
    return state


def run(state):
    case = state["case"]
    if case["call"] == "batch":
        return gb.dbscan_run_batch(state["points"], state["offsets"], state["dims"], state["eps"], state["min_pts"],
                                   mode=case["mode"], algo=case["algo"], core_out=state["core"])
    if case["call"] == "multi":
        return gb.dbscan_run_multi(state["points"], state["eps"], state["min_pts"], mode=case["mode"],
                                   algo=case["algo"], want_core=True)
    if case["call"] == "host":
        return gb.dbscan_run_host(state["points"], state["eps"], state["min_pts"][0], mode=case["mode"],
                                  algo=case["algo"], labels_out=state["labels"], core_out=state["core"])
    return gb.dbscan_run(state["points"], state["eps"], state["min_pts"][0], mode=case["mode"], algo=case["algo"],
                         want_core=True)


def work(case):
    """The coordinates read once, a label and a core flag written per point (and minPts of a sweep). The distance
    tests that decide them depend on the data and the index: none of them are counted."""
    if case["call"] == "batch":
        sizes, dims, _, _ = _instances(case)
        return {"bytes": int((sizes * dims).sum()) * 4 + int(sizes.sum()) * 5, "flops": 0}
    return {"bytes": case["n"] * (4 * case["dim"] + 5 * len(_min_pts(case))), "flops": 0}
