"""The output's order on groups of identical points around the length from
which their edges (one run of equal weight and smaller id per group) take the
three-key sort, against the oracle, bit-exact.  With options given, so that
every size takes the general path."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("morton_bits", [0, 128])
@pytest.mark.parametrize("size", [2, 33, 64, 65, 66, 67, 130, 900])
def test_groups(size, morton_bits):
    import paper_2207_00514_gb300 as pkg
    rng = np.random.default_rng(size)
    pts = synth.uniform(5000, 3, size)
    for _ in range(3):  # groups spread over the input order
        pts[rng.choice(5000, size, replace=False)] = rng.random(3).astype(np.float32)
    edges, _ = pkg.emst_compute_ex(torch.from_numpy(pts).cuda(), morton_bits=morton_bits)
    torch.cuda.synchronize()
    got = pkg.edges_numpy(edges).view(np.uint32).reshape(-1, 3)
    assert np.array_equal(got, oracle.emst(pts).view(np.uint32).reshape(-1, 3))
