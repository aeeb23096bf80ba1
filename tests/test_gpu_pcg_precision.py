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
