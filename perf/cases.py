"""The work that is timed: calls of the library's public entry points over the sizes,
shapes and options it is used with.

A case is a dict of plain values; ``prepare`` draws its inputs on the GPU from a seed,
``run`` makes one pass and returns everything the call returns.  The point sets are the
shapes the repository's own workloads have: uniform points, 2D and 3D blobs, NFW halos,
lattices with exact ties, and clusters denser than the 64-bit curve grid resolves.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2207_00514_gb300 as emst


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a few hundred 2D points, as a tool calls it in a loop: latency and launches only
        dict(name="emst_2d_333", kind="emst", dim=2, shape="blobs", n=333),
        # the 10,000-point uniform cloud: a small problem solved once
        dict(name="emst_3d_10k", kind="emst", dim=3, shape="uniform", n=10_000),
        # 1M clustered 2D points (maps, trajectories)
        dict(name="emst_2d_1m", kind="emst", dim=2, shape="blobs", n=1_000_000),
        # the benchmark's cosmology-shaped cloud at its full size
        dict(name="emst_3d_37m", kind="emst", dim=3, shape="halos", n=37_000_000),
        # points and edges in pinned host memory, read and written by the call itself
        dict(name="emst_3d_host_3m", kind="emst_host", dim=3, shape="halos", n=3_000_001),
        # quantised coordinates: many exact ties and repeated points
        dict(name="emst_3d_lattice_1m", kind="emst", dim=3, shape="lattice", n=1_000_003),
        # clusters below the 64-bit grid (GPS traces): the automatic 128-bit codes
        dict(name="emst_3d_dense_2m", kind="emst", dim=3, shape="dense", n=2_000_000),
        # many instances of very uneven size in one call
        dict(name="batch_mixed_256", kind="batched", dim=3, instances=256, lo=100, hi=1_000_000,
             layout=4),
        # many small instances in one call (one tree per object, per tile, per event)
        dict(name="batch_small_1500", kind="batched", dim=3, instances=1500, lo=100, hi=4_000,
             layout=5),
        # the clustering pipeline: mutual-reachability tree, then its dendrogram
        dict(name="hdbscan_300k_k8", kind="hdbscan", dim=3, shape="halos", n=300_007, k=8),
        # core distances alone (density estimates, outlier scores)
        dict(name="core_200k_k16", kind="core", dim=3, shape="halos", n=200_003, k=16),
        # the single-linkage hierarchy of a tree that is already there
        dict(name="dendrogram_8m", kind="dendrogram", dim=3, shape="halos", n=8_000_000),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["emst", "emst", "emst", "emst", "emst_host", "batched", "batched",
                       "hdbscan", "core", "dendrogram"])
    dim = rng.choice([2, 3])
    if kind == "batched":
        instances = _log_size(rng, 3, 2_000)
        lo = _log_size(rng, 2, 400)
        # the expected number of points stays within the listed batch's
        hi = _log_size(rng, 2 * lo, max(4 * lo, min(1_000_000, 40_000_000 // instances)))
        return dict(kind=kind, dim=dim, instances=instances, lo=lo, hi=hi,
                    layout=rng.randrange(1 << 30))
    shapes = ["uniform", "blobs", "blobs", "lattice", "dense"] + (["halos"] * 3 if dim == 3 else [])
    shape = rng.choice(shapes)
    top = {"dense": 4_000_000, "lattice": 4_000_000}.get(shape, 20_000_000)
    if kind == "hdbscan":
        shape = "blobs" if shape in ("lattice", "dense") else shape
        return dict(kind=kind, dim=dim, shape=shape, n=_log_size(rng, 200, 5_000_000),
                    k=rng.randint(2, 16))
    if kind == "core":
        shape = "uniform" if shape in ("lattice", "dense") else shape
        return dict(kind=kind, dim=dim, shape=shape, n=_log_size(rng, 200, 5_000_000),
                    k=rng.randint(2, 32))
    if kind == "dendrogram":
        return dict(kind=kind, dim=dim, shape=shape, n=_log_size(rng, 200, min(top, 10_000_000)))
    if kind == "emst_host":
        return dict(kind=kind, dim=dim, shape=shape, n=_log_size(rng, 200, min(top, 5_000_000)))
    return dict(kind=kind, dim=dim, shape=shape, n=_log_size(rng, 50, top))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _finish(x, g):
    """Rows shuffled, wrapped into the unit box, in FP32."""
    x = x[torch.randperm(x.shape[0], generator=g, device="cuda")]
    x = torch.remainder(x, 1.0).to(torch.float32)
    return torch.where(x >= 1.0, torch.zeros_like(x), x).contiguous()


def _clusters(n, dim, g, host, n_clusters, sigma_lo, sigma_hi, weights):
    """90 % of the points in Gaussian clusters, 10 % uniform."""
    n_bg = int(round(0.1 * n))
    counts = host.multinomial(n - n_bg, weights / weights.sum())
    which = torch.repeat_interleave(torch.arange(n_clusters, device="cuda"),
                                    torch.from_numpy(counts).cuda())
    centres = _rand(g, n_clusters, dim)
    sigma = torch.exp(math.log(sigma_lo) +
                      (math.log(sigma_hi) - math.log(sigma_lo)) * _rand(g, n_clusters))
    x = centres[which] + sigma[which, None] * _randn(g, n - n_bg, dim)
    return _finish(torch.cat([x, _rand(g, n_bg, dim)]), g)


def _halos(n, g, host):
    """80 % of the points in NFW halos (member counts p(m) ~ m^-1.9 on [10, 1e5]), 20 % uniform."""
    n_bg = int(round(0.2 * n))
    n_cl = n - n_bg
    sizes = []
    used = 0
    while used < n_cl:
        u = host.random(n_cl // 100 + 64)
        m = np.floor((10.0 ** -0.9 + u * (1e5 ** -0.9 - 10.0 ** -0.9)) ** (1.0 / -0.9))
        m = np.maximum(m.astype(np.int64), 1)
        sizes.append(m)
        used += int(m.sum())
    sizes = np.concatenate(sizes)
    ends = np.cumsum(sizes)
    last = int(np.searchsorted(ends, n_cl))
    sizes = sizes[:last + 1].copy()
    sizes[last] -= int(ends[last]) - n_cl
    c = 5.0
    # radius from the enclosed mass, tabulated against sqrt(mass) (smooth at the centre)
    xs = torch.linspace(0.0, 1.0, 65537, device="cuda", dtype=torch.float64) ** 2 * c
    s = torch.sqrt(torch.log1p(xs) - xs / (1.0 + xs))
    q = torch.sqrt(_rand(g, n_cl) * s[-1] ** 2)
    k = torch.searchsorted(s, q).clamp(1, 65536)
    x = xs[k - 1] + (xs[k] - xs[k - 1]) * (q - s[k - 1]) / (s[k] - s[k - 1])
    count = torch.from_numpy(sizes).cuda()
    which = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), count)
    r_vir = 0.01 * (count.to(torch.float64) / 1e5) ** (1.0 / 3.0)
    v = _randn(g, n_cl, 3)
    v /= v.norm(dim=1, keepdim=True).clamp_min(1e-300)
    pts = _rand(g, len(sizes), 3)[which] + (x / c * r_vir[which])[:, None] * v
    return _finish(torch.cat([pts, _rand(g, n_bg, 3)]), g)


def _lattice(n, dim, g):
    """Lattice sites, 96 % of them taken, and 4 % repeated points."""
    n_dup = int(0.04 * n)
    side = max(2, math.ceil(((n - n_dup) / 0.96) ** (1.0 / dim)))
    site = torch.randperm(side ** dim, generator=g, device="cuda")[:n - n_dup]
    again = torch.randint(0, n - n_dup, (n_dup,), generator=g, device="cuda")
    site = torch.cat([site, site[again]])
    site = site[torch.randperm(n, generator=g, device="cuda")]
    k = torch.stack([(site // side ** d) % side for d in range(dim)], dim=1)
    return (k.to(torch.float64) / side).to(torch.float32).contiguous()


def _points(shape, n, dim, seed):
    g = _generator(seed)
    host = np.random.default_rng(seed)
    if shape == "uniform":
        return _finish(_rand(g, n, dim), g)
    if shape == "blobs":
        return _clusters(n, dim, g, host, 50, 1e-3, 5e-2, host.dirichlet(np.ones(50)))
    if shape == "dense":
        k = max(20, min(20_000, n // 100))
        return _clusters(n, dim, g, host, k, 1e-9, 1e-6, 1.0 / (1.0 - host.random(k)))
    if shape == "lattice":
        return _lattice(n, dim, g)
    return _halos(n, g, host)


def _sizes(case):
    host = np.random.default_rng(case["layout"])
    s = np.exp(host.uniform(math.log(case["lo"]), math.log(case["hi"]), case["instances"]))
    return np.floor(s).astype(np.int64)


def _batch(case, seed):
    """Every instance: 20 blobs and 10 % uniform points, drawn for all of them at once."""
    sizes = _sizes(case)
    offsets = np.zeros(len(sizes) + 1, dtype=np.int64)
    offsets[1:] = np.cumsum(sizes)
    g = _generator(seed)
    dim, count, total = case["dim"], len(sizes), int(offsets[-1])
    which = torch.repeat_interleave(torch.arange(count, device="cuda"),
                                    torch.from_numpy(sizes).cuda())
    centres = _rand(g, count, 20, dim)
    sigma = torch.exp(math.log(1e-3) + math.log(50.0) * _rand(g, count, 20))
    blob = torch.randint(0, 20, (total,), generator=g, device="cuda")
    x = centres[which, blob] + sigma[which, blob][:, None] * _randn(g, total, dim)
    x = torch.where((_rand(g, total) < 0.1)[:, None], _rand(g, total, dim), x)
    x = torch.remainder(x, 1.0).to(torch.float32)
    return torch.where(x >= 1.0, torch.zeros_like(x), x).contiguous(), offsets


def prepare(case, seed):
    state = dict(case)
    if case["kind"] == "batched":
        state["points"], state["offsets"] = _batch(case, seed)
        return state
    pts = _points(case["shape"], case["n"], case["dim"], seed)
    if case["kind"] == "emst_host":
        state["points"] = pts.cpu().pin_memory()
    elif case["kind"] == "dendrogram":
        state["edges"] = emst.emst_compute(pts)
    else:
        state["points"] = pts
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind in ("emst", "emst_host"):
        return emst.emst_compute(state["points"])
    if kind == "batched":
        edges, offsets = emst.emst_compute_batched(state["points"], state["offsets"])
        return edges, offsets
    if kind == "hdbscan":
        edges, _ = emst.emst_compute_ex(state["points"], mrd_k=state["k"])
        linkage, parent = emst.emst_dendrogram(edges)
        return edges, linkage, parent
    if kind == "core":
        return emst.emst_core_distances(state["points"], state["k"])
    if kind == "dendrogram":
        linkage, parent = emst.emst_dendrogram(state["edges"])
        return linkage, parent
    raise ValueError(kind)


def work(case):
    """Inputs read once, outputs written once; 3 dim - 1 operations per weight that is returned."""
    dim, kind = case["dim"], case["kind"]
    per_weight = 3 * dim - 1
    if kind == "batched":
        s = _sizes(case)
        n, m = int(s.sum()), int(np.maximum(s - 1, 0).sum())
        return {"bytes": 4 * dim * n + 12 * m + 16 * (len(s) + 1), "flops": per_weight * m}
    n = case["n"]
    m = n - 1
    tree = {"bytes": 4 * dim * n + 12 * m, "flops": per_weight * m}
    hierarchy = 16 * m + 4 * (2 * n - 1)
    if kind == "hdbscan":
        return {"bytes": tree["bytes"] + hierarchy, "flops": tree["flops"] + per_weight * n * (case["k"] - 1)}
    if kind == "core":
        return {"bytes": 4 * dim * n + 4 * n, "flops": per_weight * n * (case["k"] - 1)}
    if kind == "dendrogram":
        return {"bytes": 12 * m + hierarchy, "flops": 0}
    return tree


def exact(case, seed):
    """The core distances from all pairs in FP64.  The other outputs are ids, counts and the
    bits of weights in integer tensors: there is nothing to round."""
    if case["kind"] != "core" or case["n"] > 250_000:
        return None
    x = _points(case["shape"], case["n"], case["dim"], seed).to(torch.float64)
    out = torch.empty(case["n"], dtype=torch.float64, device="cuda")
    step = max(1, (1 << 28) // case["n"])
    for a in range(0, case["n"], step):
        d = torch.zeros(min(step, case["n"] - a), case["n"], dtype=torch.float64, device="cuda")
        for q in range(case["dim"]):
            d += (x[a:a + step, q, None] - x[None, :, q]) ** 2
        out[a:a + step] = d.topk(case["k"], dim=1, largest=False).values[:, -1]
    return out
