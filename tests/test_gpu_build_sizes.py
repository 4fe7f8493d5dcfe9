"""The build (curve order, hierarchy, boxes) against the oracle at the sizes
where its parts end: the sort's tile shapes and their last tiles; the
hierarchy's CTAs of 128 chunks, the groups of 16 and 64 of them that merge, the
last merge of at most 64, and inputs that leave many splits open.  Everything is
compared exactly."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def build(pts, **kw):
    import paper_2207_00514_gb300 as pkg
    out = pkg.emst_build_bvh(torch.from_numpy(np.ascontiguousarray(pts)).cuda(), **kw)
    torch.cuda.synchronize()
    return out


# tiles of 1,024 keys up to 307,200, of 2,048 up to 614,400, of 3,584 beyond
@pytest.mark.parametrize("n", [2, 255, 1023, 1024, 1025, 307_199, 307_200, 307_201, 614_400, 614_401,
                               172 * 3584, 172 * 3584 + 1])
def test_order(n):
    pts = synth.uniform(n, 2, n)
    pts[::3] = np.round(pts[::3] * 64) / 64  # equal codes: the order has to be stable
    out = build(pts)
    lo, hi, _ = oracle.scene_box(pts)
    codes = oracle.morton(pts, lo, hi)
    perm = oracle.sort_perm(codes)
    assert np.array_equal(out["perm"].cpu().numpy().view(np.uint32), perm)
    assert np.array_equal(out["codes"].cpu().numpy().view(np.uint64), codes[perm])


def log_uniform(n, dim, seed):
    """Distances from one corner spread over all scales: long one-sided trees."""
    rng = np.random.default_rng(seed)
    return np.exp2(-22.0 * rng.random((n, dim))).astype(np.float32)


@pytest.mark.parametrize("n,make,kw", [
    *[(n, synth.blobs, {}) for n in (3, 127, 128, 129, 130, 256, 2049, 8192, 8193, 131_072, 131_073)],
    (300_001, lambda n, d, s: synth.halos(n, s), {}),
    (100_000, log_uniform, {}),
    (100_000, log_uniform, dict(morton_bits=128)),
    (50_001, lambda n, d, s: np.zeros((n, d), np.float32), {}),
    (70_000, lambda n, d, s: synth.dense(n, d, s, n_clusters=50), dict(morton_bits=128)),
    (40_003, synth.blobs, dict(leaf_size=4)),
    (2_097_153, synth.uniform, {}),
])
def test_tree(n, make, kw):
    pts = make(n, 3, n)
    leaf = kw.get("leaf_size", 1)
    out = build(pts, **kw)
    ref = oracle.bvh_reference(pts, morton_bits=kw.get("morton_bits", 64))
    codes = ref["sorted_codes"][::leaf]
    tree = oracle.radix_tree128(codes[:, 0], codes[:, 1]) if codes.ndim == 2 else oracle.radix_tree(codes)
    left, right, first, last = tree
    nc = len(codes)
    ch = out["children"].cpu().numpy().view(np.uint32).astype(np.int64)
    ch = np.where(ch & 0x80000000, (nc - 1) + (ch & 0x7FFFFFFF), ch)
    assert np.array_equal(ch[:, 0], left) and np.array_equal(ch[:, 1], right)
    boxes = out["boxes"].cpu().numpy()
    if leaf == 1:  # the oracle's own node boxes; a leaf's box is its point
        lo, hi, sp = ref["box_lo"], ref["box_hi"], ref["sorted_points"]
        for side, refs in ((0, left), (1, right)):
            inner = refs < nc - 1
            assert np.array_equal(boxes[inner, side, :3], lo[refs[inner]])
            assert np.array_equal(boxes[inner, side, 3:], hi[refs[inner]])
            at = sp[refs[~inner] - (nc - 1)]
            assert np.array_equal(boxes[~inner, side, :3], at) and np.array_equal(boxes[~inner, side, 3:], at)
