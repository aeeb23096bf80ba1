"""How far off the preconditioner of the PCG measure is where the capacitance matrix is badly conditioned (off-tree edges
that outweigh the tree up to 10^6 times): no further than the same formula in plain FP64 with the matrix inverted pivot by
pivot.  Both are FP64 evaluations of one expression whose sums differ in order alone, so the bound is four times that
one's residual, in the geometric mean over ten problems."""
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


def _star(n, m, lo, hi, seed):
    """A star of tree weights U[1,2] with m edges between leaves of weights 10^lo .. 10^hi."""
    rng = np.random.default_rng(seed)
    a, b = np.triu_indices(n, 1)
    pick = rng.choice(np.flatnonzero(a > 0), size=m, replace=False)
    u = np.concatenate([np.zeros(n - 1, dtype=np.int64), a[pick]])
    v = np.concatenate([np.arange(1, n), b[pick]])
    w = np.concatenate([1.0 + rng.random(n - 1), 10.0 ** rng.uniform(lo, hi, m)])
    order = np.lexsort((v, u))
    rp, col, cw = W.csr_from_edges(n, u[order].astype(np.int32), v[order].astype(np.int32), w[order])
    parent = np.zeros(n, dtype=np.int32)
    parent[0] = -1
    return W.Graph(n=n, row_ptr=rp, col=col, w=cw, parent=parent, name="star")


def _plain(n, u, v, w, b):
    """Grounded L_P^-1 b of the star plus the edges that miss vertex 0, by the capacitance matrix, in FP64."""
    tree = u == 0
    r = np.zeros(n)
    r[v[tree]] = 1.0 / w[tree]
    a, c, x = u[~tree], v[~tree], w[~tree]
    k = a.size
    U = np.zeros((n, k))
    U[a, np.arange(k)], U[c, np.arange(k)] = 1.0, -1.0
    C = U.T @ (r[:, None] * U) + np.diag(1.0 / x)
    for p in range(k):
        d = 1.0 / C[p, p]
        row, f = C[p] * d, C[:, p].copy()
        row[p] = d
        C[:, p] = 0.0
        rest = np.arange(k) != p
        C[rest] -= np.outer(f[rest], row)
        C[p] = row
    t = r * b
    return t - r * (U @ (C @ (t[a] - t[c])))


def _residual(n, u, v, w, z, b):
    d = w.astype(np.longdouble) * (z.astype(np.longdouble)[u] - z.astype(np.longdouble)[v])
    y = np.zeros(n, dtype=np.longdouble)
    np.add.at(y, u, d)
    np.subtract.at(y, v, d)
    return float(np.abs(y - b)[1:].max() / np.abs(b).max())


@pytest.mark.parametrize("n,m", [(130, 95), (200, 300)])
@pytest.mark.parametrize("lo,hi", [(0, 3), (3, 3), (5, 6)])
def test_heavy_edges(B, n, m, lo, hi):
    here, plain = [], []
    for seed in range(10):
        g = _star(n, m, lo, hi, seed)
        ids = O.offtree_scores(g, c=0)["id"]
        b = np.random.default_rng([seed, 1]).standard_normal(n)
        z = B.pcg_trace(g, ids, b, tol=1e-3, max_iter=1)[3]
        eu, ev, ew = g.edges()
        bb = b - b.mean()
        here.append(np.log(_residual(n, eu, ev, ew, np.asarray(z), bb)))
        plain.append(np.log(_residual(n, eu, ev, ew, _plain(n, eu, ev, ew, bb), bb)))
    assert np.mean(here) <= np.mean(plain) + np.log(4.0), (np.exp(np.mean(here)), np.exp(np.mean(plain)))


def _tour(g):
    """The Euler tour as arrays: down?, vertex, entry and exit positions, weight of the edge above."""
    n, parent = g.n, np.asarray(g.parent)
    row = np.repeat(np.arange(n), np.diff(g.row_ptr))
    above = parent[row] == g.col
    w = np.ones(n)
    w[row[above]] = g.w[above]
    kids = [[] for _ in range(n)]
    for v in np.flatnonzero(parent >= 0):
        kids[parent[v]].append(int(v))
    root = int(np.flatnonzero(parent < 0)[0])
    tour, stack = [], [(root, 0)]
    while stack:
        v, i = stack.pop()
        if i < len(kids[v]):
            stack += [(v, i + 1), (kids[v][i], 0)]
            tour.append(kids[v][i])
        elif v != root:
            tour.append(~v)
    tour = np.array(tour)
    down = tour >= 0
    v = np.where(down, tour, ~tour)
    tin, tout = np.zeros(n, dtype=np.int64), np.zeros(n, dtype=np.int64)
    tin[v[down]], tout[v[~down]] = np.flatnonzero(down), np.flatnonzero(~down)
    return down, v, tin, tout, w, root


def test_tree_solves(B):
    """The tree alone, on meshes whose weights span 10^6: the residual against that of running sums over the tour in FP64,
    one position after the other, over 81 problems.  In a model of the kernels' order of additions the ratio of the
    geometric means is 1.3 where a tile's sum is added up as its prefixes are, 1.9 where it is added up otherwise (then
    each tile's prefixes miss the next one's by that difference): the bound is 1.6."""
    here, plain = [], []
    for seed in range(1, 28):
        g = W.mesh3d_graph(8 + seed % 9, seed=seed)
        down, v, tin, tout, w, root = _tour(g)
        up = np.flatnonzero(g.parent >= 0)
        eu, ev, ew = up, g.parent[up], w[up]

        def residual(z, b):
            z = z.astype(np.longdouble)
            d = ew * (z[eu] - z[ev])
            y = np.zeros(g.n, dtype=np.longdouble)
            np.add.at(y, eu, d)
            np.subtract.at(y, ev, d)
            y -= b
            y[root] = 0
            return float(np.abs(y).max() / np.abs(b).max())

        for q in range(3):
            b = np.random.default_rng([q, seed]).standard_normal(g.n)
            bb = b - b.mean()
            here.append(np.log(residual(np.asarray(B.pcg_trace(g, np.zeros(0, np.int32), b, max_iter=1)[3]), bb)))
            E = np.concatenate([[0.0], np.cumsum(np.where(down, bb[v], 0.0))[:-1]])
            f = (E[tout] - E[tin]) / w
            x = np.cumsum(np.where(down, f[v], -f[v]))[tin]
            x[root] = 0.0
            plain.append(np.log(residual(x - x.mean(), bb)))
    assert np.mean(here) <= np.mean(plain) + np.log(1.6), np.exp(np.mean(here) - np.mean(plain))
