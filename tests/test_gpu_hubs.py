"""Trees with hubs: rows of the tree's adjacency on either side of what a thread, a block's runs of 32 and its merges
take, and hubs of 10^5 neighbours, whose rows fill in no order.  Recoveries against the oracle; the PCG measure by its
residual (z within 1e-10 of the largest entry of the exact solution, so |L_P z - b'| <= 1e-10 |L_P|_inf |z|_inf) and by
equal bits on a second run (its sums follow the rows' order)."""
from __future__ import annotations

import time

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


def _hubs(rows, seed, extra):
    """A root, below it one hub per entry of `rows` with that many tree neighbours, leaves on them, and `extra` random
    edges between leaves; vertex ids in random order."""
    rng = np.random.default_rng(seed)
    hub = np.arange(1, len(rows) + 1)
    kids = np.repeat(hub, np.asarray(rows) - 1)
    n = 1 + len(rows) + kids.size
    parent = np.concatenate([[-1], np.zeros(len(rows), dtype=np.int64), kids])
    leaf = np.arange(1 + len(rows), n)
    more = rng.choice(leaf, size=(2, extra))
    u = np.concatenate([parent[1:], more[0]])
    v = np.concatenate([np.arange(1, n), more[1]])
    perm = rng.permutation(n)
    pairs = np.unique(np.sort(np.stack([perm[u], perm[v]])[:, u != v], axis=0).T, axis=0)
    ew = np.power(10.0, rng.uniform(-3, 3, len(pairs)))
    rp, col, w = W.csr_from_edges(n, pairs[:, 0].astype(np.int32), pairs[:, 1].astype(np.int32), ew)
    p = np.full(n, -1, dtype=np.int32)
    p[perm[1:]] = perm[parent[1:]]
    return W.Graph(n=n, row_ptr=rp, col=col, w=w, parent=p, name=f"hubs{max(rows)}")


def _recoveries(B, g, k):
    _, oids, osc, _ = O.recover(g, 0.0, c=2, k_override=k)
    with B.Sparsifier.from_graph(g, options=B.default_options(k_override=k)) as sp:
        _, ids, sc, _ = sp.recover(0.0, 2, capacity=max(k, 1))
    assert np.array(ids).tolist() == oids.tolist() and np.array_equal(np.array(sc), osc)


def _residual(B, g, ids, b):
    z = [B.pcg_trace(g, ids, b, tol=1e-12, max_iter=1)[3] for _ in range(2)]
    assert np.array_equal(z[0], z[1])
    z = z[0]
    row = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    up = row < g.col
    eu, ev, ew = row[up], g.col[up], g.w[up]
    keep = (g.parent[eu] == ev) | (g.parent[ev] == eu)
    keep[ids] = True
    eu, ev, ew = eu[keep], ev[keep], ew[keep]
    d = ew * (z[eu] - z[ev])
    y, degree = np.zeros(g.n), np.zeros(g.n)
    for at, x in ((eu, d), (ev, -d)):
        np.add.at(y, at, x)
    for at in (eu, ev):
        np.add.at(degree, at, ew)
    off = np.abs(y - (b - b.mean()))
    off[g.parent < 0] = 0.0
    assert off.max() <= 1e-10 * 2 * degree.max() * np.abs(z).max()


@pytest.mark.parametrize("rows", [[63, 64, 65, 66], [95, 96, 97, 127, 128, 129, 2, 3], [255, 256, 257, 1024, 1025, 5000]])
def test_row_lengths(B, rows):
    g = _hubs(rows, seed=len(rows), extra=4 * sum(rows))
    _recoveries(B, g, min(g.n_offtree, 3000))
    off = O.offtree_scores(g, c=0)["id"]
    rng = np.random.default_rng(1)
    _residual(B, g, rng.choice(off, size=min(300, off.size), replace=False).astype(np.int32), rng.standard_normal(g.n))


@pytest.mark.parametrize("leaves", [10_000, 100_000])
def test_star(B, leaves):
    """One hub with all leaves but a few.  Sorted by one thread, the larger row alone took minutes."""
    g = _hubs([leaves, 3], seed=leaves, extra=leaves)
    t = time.perf_counter()
    with B.Sparsifier.from_graph(g):
        pass
    assert time.perf_counter() - t < 20
    _recoveries(B, g, 300)
    off = O.offtree_scores(g, c=0)["id"]
    _residual(B, g, off[::max(1, off.size // 200)][:200].astype(np.int32), np.random.default_rng(2).standard_normal(g.n))


@pytest.mark.parametrize("k", [64, 65, 3000])
def test_recovered_edges_at_one_vertex(B, k):
    """A star whose first leaf is joined to k others: the measure's list of recovered edges at that leaf has k entries."""
    n, rng = k + 40, np.random.default_rng(k)
    u = np.concatenate([np.zeros(n - 1, dtype=np.int64), np.ones(k, dtype=np.int64)])
    v = np.concatenate([np.arange(1, n), np.arange(2, k + 2)])
    perm = rng.permutation(n)
    pairs = np.sort(np.stack([perm[u], perm[v]]), axis=0).T
    pairs = pairs[np.lexsort((pairs[:, 1], pairs[:, 0]))]
    rp, col, w = W.csr_from_edges(n, pairs[:, 0].astype(np.int32), pairs[:, 1].astype(np.int32),
                                  1.0 + 9.0 * rng.random(len(pairs)))
    p = np.full(n, perm[0], dtype=np.int32)
    p[perm[0]] = -1
    g = W.Graph(n=n, row_ptr=rp, col=col, w=w, parent=p, name="joined leaf")
    off = O.offtree_scores(g, c=0)["id"]
    assert off.size == k
    _residual(B, g, rng.permutation(off).astype(np.int32), rng.standard_normal(n))
