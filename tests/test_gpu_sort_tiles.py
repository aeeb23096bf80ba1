"""The order of few candidates (tiles of 2048 sorted apart, then ranked against each other): candidate counts on either
side of one and several tiles, with many equal scores, against the oracle; the other sort gives the same."""
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


def _tied(side, seed):
    """A grid whose weights are 1 or 2: few distinct scores."""
    g = W.grid_graph(side)
    eu = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    up = eu < g.col
    eu, ev = eu[up].astype(np.int32), g.col[up]
    ew = np.random.default_rng(seed).choice([1.0, 2.0], size=eu.size)
    rp, col, w = W.csr_from_edges(g.n, eu, ev, ew)
    return W.Graph(n=g.n, row_ptr=rp, col=col, w=w, parent=W.max_spanning_tree_parent(g.n, eu, ev, ew), name="tied")


@pytest.mark.parametrize("tied", [False, True])
@pytest.mark.parametrize("k", [0, 1, 20, 1340, 1343, 1344, 1345, 1360, 2710, 4100, 12000, 21000])
def test_counts_around_tiles(B, k, tied):
    g = _tied(170, 3) if tied else W.grid_graph(170)
    _, oids, osc, _ = O.recover(g, (k + 0.5) / g.n, c=2)
    seen = []
    for one_launch in (1, 0):
        o = B.default_options(sort_one_launch=one_launch)
        with B.Sparsifier.from_graph(g, options=o) as sp:
            for _ in range(2):  # 3 k candidates first, then what did
                st, ids, sc, _ = sp.recover((k + 0.5) / g.n, 2, capacity=g.m)
                assert np.array(ids).tolist() == oids.tolist() and np.array_equal(np.array(sc), osc)
                seen.append(sp.last_stats()["candidates"])
    assert seen[:2] == seen[2:]


@pytest.mark.parametrize("factor", [1.5, 2.0, 4.0])
def test_counts_of_a_mesh(B, factor):
    g = W.mesh3d_graph(40, seed=6)
    _, oids, osc, _ = O.recover(g, 0.2, c=3)
    with B.Sparsifier.from_graph(g, options=B.default_options(candidate_factor=factor)) as sp:
        st, ids, sc, _ = sp.recover(0.2, 3, capacity=g.m)
        assert np.array(ids).tolist() == oids.tolist() and np.array_equal(np.array(sc), osc)
