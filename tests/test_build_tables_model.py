"""The build's rule and its order of work, modelled on the CPU, against the
oracle's radix tree.

The GPU builds the tree without a climb: the node of split s covers the chunks
between the nearest splits of smaller delta (the leading bits that the keys on
a split's two sides share) and is numbered by its right end when the delta on
its right is the larger one, else by its left end (the root: 0).  A CTA of
`tile` chunks builds every node whose two neighbours lie inside it; the splits
that stay open leave as items (the open split after a finished subtree and its
delta), a group of CTAs' items goes through tables of `table` entries, refilled
with what stays open, until one CTA has them all (`last` entries, where what
stays open always leaves room)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle


def build(keys, tile, table, last, group, max_group):
    n = len(keys)
    nodes = {}

    def delta(s):  # of the split between chunks s and s + 1
        if s < 0 or s + 1 >= n:
            return -1
        a, b = int(keys[s]), int(keys[s + 1])
        return 64 - (a ^ b).bit_length() if a != b else 64 + 32 - (s ^ (s + 1)).bit_length()

    def step(splits):
        """splits: (position, delta) around the items, one more than those.
        Builds what is closed and returns the items whose split stays open."""
        items = len(splits) - 1
        still_open = []
        for e in range(1, items + 1):
            d, p, q = splits[e][1], e, e + 1
            while p > 0 and splits[p - 1][1] > d:
                p -= 1
            while q <= items and splits[q][1] > d:
                q += 1
            if e == items or p == 0 or q > items:
                still_open.append(e)
                continue
            (left, dl), (right, dr) = splits[p - 1], splits[q]
            idx = right if dr > dl else 0 if dl < 0 else left + 1
            assert idx not in nodes, "a node built twice"
            nodes[idx] = (left + 1, splits[e][0], right)
        return still_open

    ctas = []
    for first in range(0, n, tile):
        end = min(first + tile, n)
        splits = [(s, delta(s)) for s in range(first - 1, end)]
        ctas.append([splits[e] for e in step(splits)])
    span = tile
    while len(ctas) > 1:
        size = len(ctas) if len(ctas) <= max_group else group
        merged = []
        for c in range(0, len(ctas), size):
            items = [x for cta in ctas[c:c + size] for x in cta]
            final = len(ctas) <= size
            room = last if final else table
            out, read = [], 0
            splits = [(c * span - 1, delta(c * span - 1))]
            while True:
                take = min(len(items) - read, room - (len(splits) - 1))
                splits += items[read:read + take]
                read += take
                still_open = step(splits)
                more = read < len(items)
                if more and (final or len(still_open) <= room // 2):
                    splits = [splits[0]] + [splits[e] for e in still_open]
                    assert len(splits) - 1 < room
                    continue
                out += [splits[e] for e in still_open]
                assert len(out) <= read, "more written than read"
                if not more:
                    break
                splits = [out[-1]]
            merged.append(out)
        ctas, span = merged, span * size
    assert len(ctas[0]) == 1
    return nodes


KINDS = {
    "random": lambda g, n: g.integers(0, 2**63, n, dtype=np.uint64),
    "duplicates": lambda g, n: g.integers(0, 20, n).astype(np.uint64),
    "one_code": lambda g, n: np.full(n, 5, np.uint64),
    "powers": lambda g, n: np.uint64(1) << g.integers(0, 63, n).astype(np.uint64),
    "log_uniform": lambda g, n: np.exp2(60 * g.random(n)).astype(np.uint64),
    "skewed": lambda g, n: (np.cumsum(g.integers(1, 4, n)) ** 3).astype(np.uint64),
}


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("tile,table,last,group,max_group", [(8, 16, 256, 3, 4), (2, 8, 200, 2, 2), (32, 64, 512, 4, 16)])
def test_range_queries_give_the_radix_tree(kind, tile, table, last, group, max_group):
    g = np.random.default_rng(tile * 31 + len(kind))
    for n in (2, 3, tile, tile + 1, int(g.integers(2, 700)), 700):
        keys = np.sort(KINDS[kind](g, n))
        nodes = build(keys, tile, table, last, group, max_group)
        left, right, first, last_ = oracle.radix_tree(keys)
        assert len(nodes) == n - 1
        for idx in range(n - 1):
            a, s, b = nodes[idx]
            assert (first[idx], last_[idx]) == (a, b)
            assert left[idx] == (n - 1 + s if a == s else s)
            assert right[idx] == (n - 1 + s + 1 if b == s + 1 else s + 1)
