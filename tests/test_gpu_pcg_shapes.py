"""The PCG measure at the edges of its kernels' blocks: 0 to 3 pivot blocks of 32, last blocks of 1 to 32 pivots, edges
at the root, tours of 2 to some 16 and 257 tiles, and parent links that close a cycle.  The preconditioner applied to
b' is checked by its residual: z is within 1e-10 of the largest entry of the exact solution (the bound of the other
PCG tests), so |L_P z - b'| <= 1e-10 |L_P|_inf |z|_inf at every vertex but the root."""
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


def _check(B, g, ids, b):
    ids = np.asarray(ids, dtype=np.int32)
    it, rel, hist, z = B.pcg_trace(g, ids, b, tol=1e-12, max_iter=1)
    assert it == 1 and len(hist) == 1 and rel == hist[0]
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
    assert off.max() <= 1e-10 * 2 * degree.max() * np.abs(z).max(), (g.name, ids.size, float(off.max()))
    assert abs(z.mean()) <= 1e-10 * np.abs(z).max()


@pytest.mark.parametrize("k", [0, 1, 2, 31, 32, 33, 63, 64, 65, 95, 97])
def test_pivot_blocks(B, k):
    g = W.grid_graph(23)
    off = O.offtree_scores(g, c=0)["id"]
    rng = np.random.default_rng(k)
    _check(B, g, rng.choice(off, size=k, replace=False), rng.standard_normal(g.n))


def test_edges_at_the_root(B):
    """A star's root with a path through its leaves: every tree path goes over the root, and an off-tree edge ends in
    it."""
    n = 300
    eu = np.concatenate([np.zeros(n - 1, dtype=np.int32), np.arange(1, n - 1, dtype=np.int32)])
    ev = np.concatenate([np.arange(1, n, dtype=np.int32), np.arange(2, n, dtype=np.int32)])
    rng = np.random.default_rng(5)
    rp, col, w = W.csr_from_edges(n, eu, ev, np.power(10.0, rng.uniform(-3, 3, eu.size)))
    parent = np.zeros(n, dtype=np.int32)
    parent[0], parent[2] = -1, 1  # the edge (0, 2) is off the tree
    g = W.Graph(n=n, row_ptr=rp, col=col, w=w, parent=parent, name="star")
    off = O.offtree_scores(g, c=0)["id"]
    assert 1 in off  # (0, 2)
    _check(B, g, np.unique(np.concatenate([[1], rng.choice(off, size=120, replace=False)])), rng.standard_normal(n))


@pytest.mark.parametrize("n", [2, 3, 128, 129, 130, 2049, 131072, 131073, 140000])
def test_tours(B, n):
    """Cycles of n vertices (n = 2: one edge): a tour of 2 (n - 1) positions, on either side of the tile sizes."""
    rng = np.random.default_rng(n)
    eu = np.arange(n - 1, dtype=np.int32)
    ev = eu + 1
    if n > 2:
        eu, ev = np.append(eu, 0).astype(np.int32), np.append(ev, n - 1).astype(np.int32)
    rp, col, w = W.csr_from_edges(n, eu, ev, 1.0 + 9.0 * rng.random(eu.size))
    parent = np.arange(-1, n - 1, dtype=np.int32)
    parent[n // 2 + 1:n - 1] = np.arange(n // 2 + 2, n, dtype=np.int32)  # two arms from vertex 0
    if n > 2:
        parent[n - 1] = 0
        if n == 3:
            parent[:] = [-1, 0, 0]
    g = W.Graph(n=n, row_ptr=rp, col=col, w=w, parent=parent, name=f"cycle{n}")
    off = O.offtree_scores(g, c=0)["id"] if n > 2 else np.zeros(0, dtype=np.int32)
    b = rng.standard_normal(n) if n < 1000 else np.where(np.arange(n) % 2 == 0, 1.0, -1.0)  # small potentials
    _check(B, g, off, b)


def test_parent_cycles_are_rejected(B):
    g = W.grid_graph(8)
    b = np.ones(g.n)
    par = g.parent.copy()
    x = next(v for v in range(g.n) if par[v] >= 0 and par[par[v]] >= 0)
    two = par.copy()
    two[par[x]] = x
    four = par.copy()
    square = [v for v in (0, 1, 9, 8)]
    if par[0] >= 0 and par[9] >= 0 and par[1] >= 0 and par[8] >= 0:
        for i, v in enumerate(square):
            four[v] = square[(i + 1) % 4]
    else:
        square = [54, 55, 63, 62]
        for i, v in enumerate(square):
            four[v] = square[(i + 1) % 4]
    for bad in (two, four):
        assert (bad < 0).sum() == 1
        h = W.Graph(n=g.n, row_ptr=g.row_ptr, col=g.col, w=g.w, parent=bad, name="cycle")
        with pytest.raises(B.PdgError) as e:
            B.pcg_quality(h, np.zeros(0, dtype=np.int32), b)
        assert e.value.status == B.PDG_E_NOT_A_TREE
