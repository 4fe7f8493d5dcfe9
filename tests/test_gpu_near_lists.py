"""The near lists of the plain form (every point's four nearest points from the
first round, from which the next rounds settle most points without a search)
against the oracle, bit-exact: fewer points than list entries, instances of
1 to 6 points among larger ones, exact ties at the list's end, groups of
identical points, weights that overflow, and the forms with and without lists
against each other."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def edges(pkg, pts, **kw):
    # (options given: the general path at every size)
    e, _ = pkg.emst_compute_ex(torch.from_numpy(np.ascontiguousarray(pts, dtype=np.float32)).cuda(), **kw)
    torch.cuda.synchronize()
    return pkg.edges_numpy(e).view(np.uint32).reshape(-1, 3)


@pytest.mark.parametrize("name,make", [
    ("n2", lambda: synth.uniform(2, 3, 1)), ("n3", lambda: synth.uniform(3, 2, 2)),
    ("n4", lambda: synth.uniform(4, 3, 3)), ("n5", lambda: synth.uniform(5, 3, 4)),
    ("n6", lambda: synth.uniform(6, 2, 5)), ("n127", lambda: synth.uniform(127, 3, 6)),
    ("n4097", lambda: synth.halos(4097, 7)),
    ("square_grid", lambda: np.stack(np.meshgrid(np.arange(40), np.arange(41)), -1).reshape(-1, 2)),
    ("cubic_grid", lambda: np.stack(np.meshgrid(*[np.arange(14)] * 3), -1).reshape(-1, 3)),
    ("fives", lambda: np.repeat(synth.uniform(400, 3, 8), 5, axis=0)),
    ("sixties", lambda: np.repeat(synth.uniform(30, 2, 9), 60, axis=0)),
    ("overflow", lambda: synth.uniform(300, 3, 10) * np.float32(3e25)),
])
def test_against_oracle(name, make):
    import paper_2207_00514_gb300 as pkg
    pts = np.ascontiguousarray(make(), dtype=np.float32)
    pts = pts[np.random.default_rng(3).permutation(len(pts))]
    want = oracle.emst(pts).view(np.uint32).reshape(-1, 3)
    assert np.array_equal(edges(pkg, pts), want)
    assert np.array_equal(edges(pkg, pts, carried_radius=False), want)  # without lists
    assert np.array_equal(edges(pkg, pts, count_visits=True), want)


def test_small_instances():
    import paper_2207_00514_gb300 as pkg
    sizes = [1, 2, 3, 4, 5, 6, 0, 700, 1, 5, 33, 2]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts = synth.blobs(int(offs[-1]), 3, 11)
    e, eo = pkg.emst_compute_batched(torch.from_numpy(pts).cuda(), offs)
    torch.cuda.synchronize()
    got = pkg.edges_numpy(e).view(np.uint32).reshape(-1, 3)
    for k, s in enumerate(sizes):
        if s > 1:
            want = oracle.emst(pts[offs[k]:offs[k + 1]]).view(np.uint32).reshape(-1, 3)
            assert np.array_equal(got[eo[k]:eo[k + 1]], want), s
