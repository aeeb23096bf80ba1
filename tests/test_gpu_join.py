"""The join that decides the candidates (tree cells, exact tests, settling in rank order) and the tiers it hands full
cells to, against the CPU oracle: ids and scores are compared bit for bit (whole numbers and once-rounded doubles)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from tests.helpers import graph_from_edges

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2508_20403_gb300 import binding, build

    build.build()
    binding.load()
    return binding


def _hubs(groups, seed, tail=0):
    """A root with one hub per entry (children, leaves) of `groups`; a hub's children carry the leaves, and every pair
    of leaves under different children of a hub is an edge with probability 1/2: one cell per pair of children.
    `tail` extra vertices hang below the last leaf as a path with chords to its ancestors (edges that end on their
    LCA).  Tree weights are distinct; some off-tree weights tie."""
    rng = np.random.default_rng(seed)
    edges, parent = [], [-1]

    def vertex(p):
        parent.append(p)
        edges.append((p, len(parent) - 1, 10.0 + float(rng.random())))
        return len(parent) - 1

    for children, leaves in groups:
        hub = vertex(0)
        rows = [[vertex(ch) for _ in range(leaves)] for ch in [vertex(hub) for _ in range(children)]]
        for i in range(children):
            for j in range(i):
                edges += [(a, b, float(rng.choice([1.0, 2.0, rng.random() + 0.1])))
                          for a in rows[i] for b in rows[j] if rng.random() < 0.5]
    chain = [len(parent) - 1]
    for _ in range(tail):
        chain.append(vertex(chain[-1]))
    edges += [(chain[i], chain[j], float(rng.random() + 0.5))
              for i in range(len(chain)) for j in range(i + 2, min(i + 9, len(chain)))]
    return graph_from_edges(len(parent), edges, parent, "hubs")


def _check(B, g, c, **opt):
    _, oids, osc, _ = O.recover(g, 0.0, c=c, k_override=g.n_offtree)
    with B.Sparsifier.from_graph(g, options=B.default_options(k_override=g.n_offtree, **opt)) as sp:
        for _ in range(3):  # plain, then as a later call starts (and replays)
            _, ids, sc, _ = sp.recover(0.0, c, capacity=g.m)
            assert np.array(ids).tolist() == oids.tolist(), (c, opt, sp.last_stats())
            assert np.array_equal(np.array(sc), osc)
        return sp.last_stats()


@pytest.mark.parametrize("c", [1, 2, 3])
@pytest.mark.parametrize("leaves", [2, 4, 5, 12])
def test_cell_sizes(B, c, leaves):
    """Cells of about 2, 8, 12 and 72 members: inline ones, one row and several, below the tiers' limit; chords on a
    path beside them, so that edges with an endpoint on the LCA probe too."""
    g = _hubs([(4, leaves), (3, leaves + 1)], seed=leaves, tail=40)
    stats = _check(B, g, c, use_graph=1)
    assert stats["max_subtask"] >= leaves * leaves


@pytest.mark.parametrize("c", [1, 2, 3])
@pytest.mark.parametrize("wm,bm", [(32, 0), (8, 896)])
def test_full_cells_go_to_the_tiers(B, c, wm, bm):
    """Two cells of more than 2,048 members, beside subtasks of the warp, block and cooperative tiers' sizes."""
    g = _hubs([(2, 70), (4, 12), (3, 4), (2, 3), (2, 66)], seed=7, tail=30)
    _check(B, g, c, warp_tier_max=wm, block_tier_max=bm, use_graph=1)


def test_statistics_of_the_subtasks(B):
    """Subtasks, the largest one and the candidates in subtasks of several, counted without grouping by LCA."""
    g = _hubs([(3, 6), (2, 4), (2, 1)], seed=3, tail=25)
    facts = O.offtree_scores(g, c=2)
    sizes = np.unique(facts["lca"], return_counts=True)[1]
    stats = _check(B, g, 2)
    assert stats["candidates"] == g.n_offtree
    assert (stats["subtasks"], stats["max_subtask"]) == (len(sizes), sizes.max())
    assert stats["coop_candidates"] == sizes[sizes > 1].sum()
