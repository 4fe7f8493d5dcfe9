"""The dendrogram's one-CTA form (trees of up to 4,096 edges) against the
oracle, bit-exact: at the sizes where its CTA, its threads' shares, its sort's
powers of two and the form itself end, every tree shape, with and without tied
weights, each output alone, host buffers, and what is no tree."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [2, 3, 4, 31, 32, 33, 34, 64, 65, 66, 1024, 1025, 1026, 2048, 2049, 2050, 4095, 4096, 4097, 4098]


def tensor(edges, device="cuda"):
    t = torch.from_numpy(np.ascontiguousarray(edges).view(np.int32).reshape(-1, 3).copy())
    return t.cuda() if device == "cuda" else t.pin_memory() if device == "pinned" else t


def check(edges, n, device="cuda", **kw):
    import paper_2207_00514_gb300 as pkg
    link, parent = pkg.emst_dendrogram(tensor(edges, device), n, **kw)
    torch.cuda.synchronize()
    want_link, want_parent = oracle.dendrogram(edges, n)
    if link is not None:
        got = pkg.linkage_numpy(link).view(np.uint32).reshape(-1, 4)
        assert np.array_equal(got, want_link.view(np.uint32).reshape(-1, 4)), n
    if parent is not None:
        assert np.array_equal(parent.cpu().numpy().view(np.uint32), want_parent), n


@pytest.mark.parametrize("shape", synth.TREE_SHAPES)
def test_sizes(shape):
    for n in SIZES:
        for ties in (0, 4):
            check(synth.tree_edges(n, n + ties, shape, ties=ties), n)


@pytest.mark.parametrize("device", ["pinned", "pageable"])
def test_host_buffers(device):
    check(synth.tree_edges(1500, 6, "random", ties=9), 1500, device)


def test_each_output_alone():
    e = synth.tree_edges(777, 7, "caterpillar")
    check(e, 777, parent=False)
    check(e, 777, linkage=False)


def test_not_a_tree():
    import paper_2207_00514_gb300 as pkg
    good = synth.tree_edges(500, 8, "random")

    def bad(change):
        e = good.copy()
        change(e)
        with pytest.raises(pkg.EmstError) as err:
            pkg.emst_dendrogram(tensor(e), 500)
        assert err.value.status == -1

    def cycle(e):  # the last two edges close a triangle with two vertices of the first
        e["i"][-1], e["j"][-1] = e["i"][0], e["j"][0]

    bad(cycle)
    bad(lambda e: e["i"].__setitem__(3, 500))
    bad(lambda e: e["j"].__setitem__(499 - 1, 0xFFFFFFFF))
    bad(lambda e: e["j"].__setitem__(7, e["i"][7]))
    bad(lambda e: e["w"].__setitem__(11, np.nan))
    bad(lambda e: e["w"].__setitem__(200, -1.0))
    check(good, 500)


@pytest.mark.parametrize("n", [4_500_000, 9_000_000])
def test_one_chain_over_many_tiles(n):
    # a path of rising weights is one chain: every tile of the running totals
    # continues it, found tile by tile at the one size, by the scan at the other
    check(synth.tree_edges(n, 9, "path_sorted"), n)
