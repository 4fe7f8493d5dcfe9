"""The general path at sizes that emst_compute gives to the one-launch path:
with options given every size takes it.  Whole trees against the oracle,
bit-exact, among them the output's order on runs of equal weights and the
fallback on runs too long for it; host buffers; and non-finite coordinates,
which the scene box reports (per CTA, on every way it reads the points) before
the tree that was launched meanwhile is used."""
from __future__ import annotations

import os

import numpy as np
import pytest

import oracle
import synth
from test_gpu_parity import EMST_CASES

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def words(edges):
    import paper_2207_00514_gb300 as pkg
    torch.cuda.synchronize()
    return pkg.edges_numpy(edges).view(np.uint32).reshape(-1, 3)


def want(pts):
    e = oracle.prim(pts) if len(pts) <= 4000 else oracle.kd_boruvka(pts, threads=os.cpu_count() or 4)
    return e.view(np.uint32).reshape(-1, 3)


@pytest.mark.parametrize("name,make", EMST_CASES, ids=[c[0] for c in EMST_CASES])
def test_emst_matches_oracle(name, make):
    import paper_2207_00514_gb300 as pkg
    pts = np.ascontiguousarray(make(), dtype=np.float32)
    t = torch.from_numpy(pts).cuda()
    w = want(pts)
    assert np.array_equal(words(pkg.emst_compute_ex(t)[0]), w)
    assert np.array_equal(words(pkg.emst_compute_ex(t, morton_bits=128)[0]), w)


@pytest.mark.parametrize("n,dim", [(20_000, 3), (4_999, 2), (5, 3)])
def test_host_buffers(n, dim):
    import paper_2207_00514_gb300 as pkg
    pts = synth.halos(n, 5) if dim == 3 else synth.blobs(n, 2, 5)
    w = want(pts)
    assert np.array_equal(words(pkg.emst_compute_ex(torch.from_numpy(pts).pin_memory())[0]), w)
    out = torch.empty((n - 1, 3), dtype=torch.int32)  # pageable
    pkg.emst_compute_ex(torch.from_numpy(pts.copy()), out_edges=out)
    assert np.array_equal(words(out), w)


# 3 * 1,001 and 2 * 40,001 coordinates leave a tail behind the copy's 16-byte loads
@pytest.mark.parametrize("dim,n", [(3, 1001), (2, 40_001), (3, 300_003)])
@pytest.mark.parametrize("where", ["first", "last", "last_cta", "middle"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite(dim, n, where, bad):
    import paper_2207_00514_gb300 as pkg
    pts = synth.uniform(n, dim, 3)
    at = {"first": (0, 0), "last": (n - 1, dim - 1), "last_cta": ((n - 1) // 256 * 256, 1), "middle": (n // 2, 0)}
    broken = pts.copy()
    broken[at[where]] = bad
    t = torch.from_numpy(broken)
    good = torch.from_numpy(pts).cuda()
    for points in (t.cuda(), t.pin_memory(), t):
        for kw in ({}, dict(morton_bits=64), dict(morton_bits=128)):
            with pytest.raises(pkg.EmstError) as e:
                pkg.emst_compute_ex(points, **kw)
            assert e.value.status == -2
    # the next call on the stream is not touched by it
    assert np.array_equal(words(pkg.emst_compute_ex(good)[0]), words(pkg.emst_compute(good)))


def test_non_finite_batched():
    import paper_2207_00514_gb300 as pkg
    pts = synth.uniform(9001, 3, 4)
    offsets = np.array([0, 1, 3000, 3000, 9001], dtype=np.int64)
    for row in (0, 2999, 9000):
        broken = pts.copy()
        broken[row, 2] = np.nan
        for points in (torch.from_numpy(broken).cuda(), torch.from_numpy(broken).pin_memory()):
            with pytest.raises(pkg.EmstError) as e:
                pkg.emst_compute_batched(points, offsets)
            assert e.value.status == -2
    edges, at = pkg.emst_compute_batched(torch.from_numpy(pts).cuda(), offsets)
    got = words(edges)
    for k in range(4):
        part = pts[offsets[k]:offsets[k + 1]]
        if len(part) > 1:
            assert np.array_equal(got[at[k]:at[k + 1]], want(part))


@pytest.mark.parametrize("dim", [2, 3])
def test_overflowing_weights(dim):
    # nearly all pairs weigh +inf: every search's bounds tie with its best, and
    # only the tie rule keeps it from visiting every point (4 to 60 times the
    # time of the same points closer together without it)
    import statistics
    import time

    import paper_2207_00514_gb300 as pkg
    near = np.random.default_rng(dim).normal(size=(40_000, dim)).astype(np.float32)
    far = near * np.float32(1e25)

    def median_s(points):
        t = torch.from_numpy(points).cuda()
        times = []
        for _ in range(8):
            torch.cuda.synchronize()
            a = time.perf_counter()
            edges = pkg.emst_compute(t)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - a)
        return statistics.median(times[1:]), words(edges)

    far_s, got = median_s(far)
    assert far_s < 4 * median_s(near)[0]
    # (w, i, j): all weigh +inf but the pairs close enough, so nearly all edges meet point 0
    e, _ = pkg.emst_compute_ex(torch.from_numpy(far).cuda(), traversal=2)  # another search
    assert np.array_equal(got, words(e))
    small = far[:3000]
    assert np.array_equal(words(pkg.emst_compute_ex(torch.from_numpy(small).cuda())[0]), want(small))
