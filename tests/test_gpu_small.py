"""The one-launch path of small problems (emst_compute without options, up to
32,768 points) against the oracle, bit-exact, at the sizes where its blocks of
32 points, superblocks of 1,024, sort tiles and the path itself end, on inputs
with exact ties, repeated points, clusters below the 64-bit grid and weights
that overflow FP32."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def check(pts, device="cuda"):
    import paper_2207_00514_gb300 as pkg
    t = torch.from_numpy(np.ascontiguousarray(pts, dtype=np.float32))
    t = t.cuda() if device == "cuda" else t.pin_memory() if device == "pinned" else t
    e = pkg.emst_compute(t)
    torch.cuda.synchronize()
    got = pkg.edges_numpy(e).view(np.uint32).reshape(-1, 3)
    want = oracle.emst(np.ascontiguousarray(pts, dtype=np.float32)).view(np.uint32).reshape(-1, 3)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 63, 65, 1023, 1024, 1025, 2049, 16383, 16384, 16385, 32767,
                               32768, 32769])
def test_sizes(n, dim):
    check(synth.blobs(n, dim, n) if n >= 31 else synth.uniform(n, dim, n))


@pytest.mark.parametrize("name,make", [
    ("lattice", lambda: synth.lattice_ties(15_000, 700, side=25)),
    ("one_place", lambda: np.zeros((3000, 3), np.float32)),
    ("two_places", lambda: np.repeat(np.float32([[0, 0], [1, 1]]), 700, axis=0)),
    ("line", lambda: np.stack([np.arange(4000) % 1999, np.zeros(4000)], 1).astype(np.float32)),
    ("dense", lambda: synth.dense(20_000, 3, 5, n_clusters=40)),
    # squared distances beyond FP32: edges of weight +inf, ordered by id
    ("overflow", lambda: (synth.uniform(500, 3, 3) * np.float32(3e25))),
    ("huge_extent", lambda: np.concatenate([synth.uniform(300, 2, 4), synth.uniform(40, 2, 5) * np.float32(3e38)])),
])
def test_shapes(name, make):
    check(make())


@pytest.mark.parametrize("device", ["pinned", "pageable"])
def test_host_buffers(device):
    check(synth.halos(5001, 8), device)


def test_non_finite():
    import paper_2207_00514_gb300 as pkg
    p = synth.uniform(700, 3, 1)
    for bad in (np.nan, np.inf):
        q = p.copy()
        q[699, 2] = bad
        with pytest.raises(pkg.EmstError) as e:
            pkg.emst_compute(torch.from_numpy(q).cuda())
        assert e.value.status == -2
    check(p)
