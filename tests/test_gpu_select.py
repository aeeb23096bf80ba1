"""Scoring over the whole edge list and the two-step selection (list of the boundary bucket, then the exact prefix)
against the CPU oracle, at the sizes where tiles end and where the list does not fit at first: ids and scores bit for
bit."""
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


def _ladder(m, seed):
    """A connected graph of exactly m edges: a path with chords of length 2 .. 5."""
    rng = np.random.default_rng(seed)
    n = max(8, m // 3)
    u = [np.arange(n - d) for d in range(1, 6)]
    v = [x + d for d, x in enumerate(u, 1)]
    u, v = np.concatenate(u)[:m], np.concatenate(v)[:m]
    eu, ev = W._canonical(n, u, v)
    assert eu.shape[0] == m
    return W.build_graph(n, eu, ev, 1.0 + 9.0 * rng.random(m))


@pytest.mark.parametrize("m", [31, 8191, 8192, 8193, 16385, 3 * 8192 + 1])
def test_edge_counts_at_tile_ends(B, m):
    g = _ladder(m, m)
    for k in (0, 1, max(1, g.n // 10)):
        _, oids, osc, _ = O.recover(g, 0.0, c=2, k_override=k)
        with B.Sparsifier.from_graph(g, options=B.default_options(k_override=k)) as sp:
            _, ids, sc, _ = sp.recover(0.0, 2, capacity=g.m)
        assert np.array(ids).tolist() == oids.tolist() and np.array_equal(np.array(sc), osc)


@pytest.mark.parametrize("use_graph", [0, 1])
def test_boundary_bucket_larger_than_the_list(B, use_graph):
    """Unit weights: the scores share a few exponents, so the bucket of a tiny budget holds most of the 62,000
    off-tree edges and the list (four times the candidate buffers) has to grow."""
    eu, ev = W.mesh3d_edges(32)
    g = W.build_graph(32 ** 3, eu, ev, np.ones(eu.shape[0]))
    _, oids, osc, _ = O.recover(g, 0.0, c=2, k_override=20)
    with B.Sparsifier.from_graph(g, options=B.default_options(k_override=20, use_graph=use_graph)) as sp:
        for _ in range(3):
            _, ids, sc, _ = sp.recover(0.0, 2, capacity=64)
            assert np.array(ids).tolist() == oids.tolist() and np.array_equal(np.array(sc), osc)


def test_many_small_graphs_in_one_tile(B):
    """Graphs of 30 to 3,000 edges: several graphs' edges share a tile, some graphs take their whole edge list."""
    graphs = [_ladder(m, m) for m in (30, 45, 31, 3000, 60, 200, 33, 2500, 90, 1000)] * 4
    graphs += [W.grid_graph(2, 30, seed=5), W.grid_graph(40, seed=6)]
    pk = W.pack_graphs(graphs)
    alphas = np.array([0.02, 0.1, 0.3, 0.9] * 11)[:len(graphs)]
    with B.BatchSparsifier.from_packed(pk) as bs:
        for _ in range(2):
            _, op, ids, sc, counts, _ = bs.recover_batch(alphas, c=2)
            for i, g in enumerate(graphs):
                _, oids, osc, _ = O.recover(g, float(alphas[i]), c=2)
                assert np.array(ids[op[i]:op[i] + counts[i]]).tolist() == oids.tolist(), (i, g.m)
                assert np.array_equal(np.array(sc[op[i]:op[i] + counts[i]]), osc)
