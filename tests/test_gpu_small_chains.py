"""Small problems whose components form long chains (points in order on a line,
at equal or growing distances: every point's edge leads to its neighbour), on
the one-launch path against the oracle, bit-exact, and in time against the
general path: the chains are walked point by point on both, and a CTA that
waits at a barrier must not slow the one that walks."""
from __future__ import annotations

import statistics
import time

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def line(n, growing=False):
    x = np.cumsum(np.arange(n)) if growing else np.arange(n)
    return np.stack([x, np.zeros(n)], 1).astype(np.float32)


@pytest.mark.parametrize("pts", [line(33), line(3000), line(3000)[::-1], line(4000, growing=True), line(20_000)])
def test_chains(pts):
    import paper_2207_00514_gb300 as pkg
    pts = np.ascontiguousarray(pts)
    e = pkg.emst_compute(torch.from_numpy(pts).cuda())
    torch.cuda.synchronize()
    got = pkg.edges_numpy(e).view(np.uint32).reshape(-1, 3)
    assert np.array_equal(got, oracle.emst(pts).view(np.uint32).reshape(-1, 3))


def test_waiting_leaves_the_walk_alone():
    # (walked through L2 at every step it took 2.2 times the general path's time)
    import paper_2207_00514_gb300 as pkg
    t = torch.from_numpy(line(10_000)).cuda()

    def median_us(call):
        times = []
        for _ in range(12):
            torch.cuda.synchronize()
            a = time.perf_counter()
            call()
            torch.cuda.synchronize()
            times.append(time.perf_counter() - a)
        return statistics.median(times[2:])

    assert median_us(lambda: pkg.emst_compute(t)) < 1.5 * median_us(lambda: pkg.emst_compute_ex(t))
