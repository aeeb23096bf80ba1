"""The tiers (warp, block, cooperative with its rounds and serial finisher) on graphs that the join would decide: a hub
is joined to each graph whose candidates, all in one cell and with the highest scores, send the whole set to the tiers.
Every case asserts that they decided, and compares ids and scores with the oracle bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from paper_2508_20403_gb300 import workloads as W
from tests.helpers import random_small_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2508_20403_gb300 import binding, build

    build.build()
    binding.load()
    return binding


def with_hub(g, seed=0, leaves=70):
    """g with a hub of two children and `leaves` leaves each below its root, half of the pairs of leaves of different
    children joined: 2,450 candidates in one cell of the join, which takes 2,048."""
    rng = np.random.default_rng([seed, 7])
    eu, ev, ew = g.edges()
    hub, kids = g.n, np.array([g.n + 1, g.n + 2])
    leaf = g.n + 3 + np.arange(2 * leaves).reshape(2, leaves)
    n = g.n + 3 + 2 * leaves
    root = int(np.flatnonzero(g.parent < 0)[0])
    parent = np.concatenate([g.parent, [root, hub, hub], np.repeat(kids, leaves)]).astype(np.int32)
    a, b = (x.ravel() for x in np.meshgrid(leaf[0], leaf[1], indexing="ij"))
    pick = rng.random(a.size) < 0.5
    a, b = a[pick], b[pick]
    assert a.size > 2300
    tu = np.concatenate([[root, hub, hub], np.repeat(kids, leaves)])
    tv = np.arange(g.n, n)
    u = np.concatenate([eu, tu, a]).astype(np.int32)
    v = np.concatenate([ev, tv, b]).astype(np.int32)
    w = np.concatenate([ew, np.ones(tu.size), 2.0**40 * (1.0 + rng.integers(0, 40, a.size) / 8.0)])  # ties among them
    order = np.lexsort((v, u))
    rp, col, cw = W.csr_from_edges(n, u[order], v[order], w[order])
    return W.Graph(n=n, row_ptr=rp, col=col, w=cw, parent=parent, name=g.name + "+hub")


def _compare(B, g, alpha, c=2, mode=0, k_override=None, calls=1, **opt):
    _, oids, osc, _ = O.recover(g, alpha, c=c, score_mode=mode, **({} if k_override is None else {"k_override": k_override}))
    o = B.default_options(score_mode=mode, **opt)
    if k_override is not None:
        o.k_override = k_override
    with B.Sparsifier.from_graph(g, options=o) as sp:
        for _ in range(calls):
            _, ids, sc, _ = sp.recover(alpha, c, capacity=g.m)
            assert sp.last_path() == B.PATH_TIERS
            assert np.array(ids).tolist() == oids.tolist(), (g.name, alpha, c, mode, opt, sp.last_stats())
            assert np.array_equal(np.array(sc), osc)
        return sp.last_stats()


def test_random_graphs(B):
    rng = np.random.default_rng(11)
    for i in range(40):
        g = with_hub(random_small_graph(rng, n_lo=2, n_hi=24, tree="mixed"), seed=i)
        _compare(B, g, 0.0, c=int(rng.integers(1, 4)), mode=int(rng.integers(0, 2)), k_override=g.n_offtree,
                 warp_tier_max=int(rng.choice([1, 2, 4, 32])), block_tier_max=int(rng.choice([0, 3, 8, 896])),
                 max_rounds=int(rng.choice([1, 2, 8])), candidate_factor=1.0)


@pytest.mark.parametrize("c", [1, 2, 3])
def test_rmat_full_pass(B, c):
    """Every off-tree edge, two rounds, then the serial finisher."""
    g = with_hub(W.rmat_graph(11, seed=5))
    _compare(B, g, 0.0, c=c, k_override=g.n_offtree, max_rounds=2)


@pytest.mark.parametrize("rounds", [1, 8])
def test_mesh_cooperative_only(B, rounds):
    g = with_hub(W.mesh3d_graph(48, seed=44))
    stats = _compare(B, g, 0.1, warp_tier_max=1, max_rounds=rounds, calls=2)
    assert stats["coop_candidates"] > 5000 and stats["max_subtask"] > 64


@pytest.mark.parametrize("wm,bm", [(1, 896), (32, 0), (32, 64), (8, 33), (32, 896)])
def test_block_tier_bounds(B, wm, bm):
    _compare(B, with_hub(W.mesh3d_graph(32, seed=44)), 0.1, warp_tier_max=wm, block_tier_max=bm)
    g = with_hub(W.rmat_graph(13, seed=77))
    for c in (1, 2, 3):
        stats = _compare(B, g, 0.1, c=c, warp_tier_max=wm, block_tier_max=bm)
        assert stats["max_subtask"] > 896  # beyond the block tier


@pytest.mark.parametrize("graph,c,attempts", [("grid", 2, 3), ("rmat", 3, 4)])
def test_exact_blocks_run_out(B, graph, c, attempts):
    """More flagged pairs than the pool of exact blocks holds: the attempt is repeated with four times as many (once for
    the grid, twice for R-MAT, after the join's attempt); the next recovery keeps them."""
    g = with_hub(W.grid_graph(150) if graph == "grid" else W.rmat_graph(13, seed=77))
    stats = _compare(B, g, 0.0, c=c, k_override=g.n_offtree, warp_tier_max=1)
    assert stats["attempts"] == attempts
    stats = _compare(B, g, 0.0, c=c, k_override=g.n_offtree, warp_tier_max=1, calls=3, use_graph=1)
    assert stats["attempts"] == 1


@pytest.mark.parametrize("mode", [0, 1])
def test_score_modes_and_ties(B, mode):
    eu, ev = W.grid2d_edges(20, 20)
    g = with_hub(W.build_graph(400, eu, ev, np.ones(eu.shape[0])))
    _compare(B, g, 0.0, mode=mode, k_override=g.n_offtree)


@pytest.mark.parametrize("one_launch", [0, 1])
def test_orders(B, one_launch):
    """The grouping by LCA in both forms of the sort."""
    _compare(B, with_hub(W.mesh3d_graph(32, seed=4)), 0.1, sort_one_launch=one_launch)
    _compare(B, with_hub(W.rmat_graph(13, seed=77)), 0.5, sort_one_launch=one_launch)


@pytest.mark.parametrize("use_graph", [0, 1])
def test_budgets_of_one_handle(B, use_graph):
    """The rounds of an earlier budget, replayed or not; budgets that the join decides in between."""
    g = with_hub(W.rmat_graph(13, seed=77))
    small = 20.5 / g.n
    seen = []
    with B.Sparsifier.from_graph(g, options=B.default_options(use_graph=use_graph)) as sp:
        for alpha in (0.2, 0.2, 0.5, small, 0.5, 0.2, small, small, 0.2, 0.5):
            _, oids, osc, _ = O.recover(g, alpha, c=2)
            _, ids, sc, _ = sp.recover(alpha, 2, capacity=g.m)
            assert np.array(ids).tolist() == oids.tolist(), (alpha, sp.last_stats())
            assert np.array_equal(np.array(sc), osc)
            seen.append(sp.last_path())
    assert seen[:3] == [B.PATH_TIERS] * 3


@pytest.mark.parametrize("use_graph", [0, 1])
def test_batch(B, use_graph):
    """One full cell among the graphs of a batch sends all of them to the tiers."""
    graphs = [W.batch_member(i, seed=123, n_lo=200, n_hi=3000, side_lo=5, side_hi=40) for i in range(12)]
    graphs[5] = with_hub(graphs[5])
    alphas = np.array([[0.02, 0.05, 0.30][i % 3] for i in range(len(graphs))])
    with B.BatchSparsifier.from_packed(W.pack_graphs(graphs), options=B.default_options(use_graph=use_graph)) as bs:
        for _ in range(3):
            _, op, ids, sc, cnt, _ = bs.recover_batch(alphas, c=2)
            assert bs.last_path() == B.PATH_TIERS
            for i, g in enumerate(graphs):
                _, oids, osc, _ = O.recover(g, alphas[i], c=2)
                assert ids[op[i]:op[i] + cnt[i]].tolist() == oids.tolist(), i
                assert np.array_equal(sc[op[i]:op[i] + cnt[i]], osc)
