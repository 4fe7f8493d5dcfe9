"""The build (curve order, hierarchy, boxes) against the oracle at the sizes
where its parts end: the sort's tile shapes and their last tiles.  Everything
is compared exactly."""
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
