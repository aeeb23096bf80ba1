"""The order of few candidates at exact counts: tiles of 512, 1,024 and 2,048 (chosen by the capacity), counts on either
side of one and two tiles, where a single tile needs no ranking, and the largest of each capacity, with distinct and
with equal scores.  c = 0: every candidate is recovered, so the recovered edges are the order itself."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_20403_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2508_20403_gb300 import binding, build

    build.build()
    binding.load()
    return binding


def _star(scores, leaves=700, seed=0):
    """A star with unit weights and one edge between leaves per entry of `scores`, which is its score (R_T = 2)."""
    rng = np.random.default_rng(seed)
    a, b = np.triu_indices(leaves, 1)
    pick = rng.choice(a.size, size=len(scores), replace=False)
    u = np.concatenate([np.zeros(leaves, dtype=np.int64), a[pick] + 1])
    v = np.concatenate([np.arange(1, leaves + 1), b[pick] + 1])
    w = np.concatenate([np.ones(leaves), np.asarray(scores) / 2.0])
    order = np.lexsort((v, u))
    rp, col, cw = W.csr_from_edges(leaves + 1, u[order].astype(np.int32), v[order].astype(np.int32), w[order])
    parent = np.zeros(leaves + 1, dtype=np.int32)
    parent[0] = -1
    return W.Graph(n=leaves + 1, row_ptr=rp, col=col, w=cw, parent=parent, name="star")


def _order(g):
    facts = O.offtree_scores(g, c=0)
    order = np.lexsort((facts["id"], -facts["score"]))
    return facts["id"][order], facts["score"][order]


def _recover(sp, g, order, k):
    _, ids, sc, _ = sp.recover((k + 0.5) / g.n, 0, capacity=g.m)
    assert np.array_equal(np.asarray(ids), order[0][:k]) and np.array_equal(np.asarray(sc), order[1][:k])
    return sp.last_stats()["candidates"]


CASES = [(512, 5000), (512, 8192), (1024, 8193), (1024, 20000), (1024, 32768), (2048, 32769), (2048, 65536)]


@pytest.mark.parametrize("tile,capacity", CASES)
def test_distinct_scores(B, tile, capacity):
    """Every score in a bucket of its own, so a prefix has the count that is asked for (k + 32 at factor 1)."""
    i = np.random.default_rng(tile).permutation(capacity)
    g = _star(2.0 ** (i // 4096) * (1.0 + (i % 4096) / 4096.0))
    order = _order(g)
    with B.Sparsifier.from_graph(g, options=B.default_options(candidate_factor=1.0)) as sp:
        assert _recover(sp, g, order, capacity) == capacity
        for n in (32, 33, tile - 1, tile, tile + 1, 2 * tile, 2 * tile + 1, capacity // tile * tile, capacity - 1):
            if n < capacity:
                assert _recover(sp, g, order, n - 32) == n


@pytest.mark.parametrize("tile,capacity", CASES)
def test_equal_scores(B, tile, capacity):
    """The highest `n` scores are equal, and so are all others."""
    for n in (tile - 1, tile, tile + 1, 2 * tile, 2 * tile + 1, capacity):
        high = np.random.default_rng(n).permutation(capacity) < n
        g = _star(np.where(high, 8.0, 2.0), seed=n)
        order = _order(g)
        with B.Sparsifier.from_graph(g, options=B.default_options(candidate_factor=1.0)) as sp:
            assert _recover(sp, g, order, capacity) == capacity
            assert _recover(sp, g, order, n - 40) == n
