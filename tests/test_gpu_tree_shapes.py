"""Spanning trees and the checks of a graph where their kernels change path: BFS levels narrower and wider than a
queue holds, rows that a whole block shares (more of them than one block lists), lists of 1 to 70 arcs and many
components, runs of empty rows, entries without a mirror image on either side of the diagonal."""
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


def _graph(n, eu, ev, ew, name):
    eu, ev = np.minimum(eu, ev).astype(np.int32), np.maximum(eu, ev).astype(np.int32)
    rp, col, w = W.csr_from_edges(n, eu, ev, np.asarray(ew, dtype=np.float64))
    return W.Graph(n=n, row_ptr=rp, col=col, w=w, parent=np.full(n, -1, dtype=np.int32), name=name)


def _burst(hubs, leaves, tail, rng):
    """A root with `hubs` neighbours and 400 more, `leaves` leaves on each, then a path: the frontier is narrow, wide
    and narrow again."""
    eu, ev, nxt = [], [], 1
    hub = list(range(1, hubs + 1))
    nxt += hubs
    for h in hub:
        eu.append(0), ev.append(h)
    for _ in range(400):
        eu.append(0), ev.append(nxt)
        nxt += 1
    for h in hub:
        for _ in range(leaves):
            eu.append(h), ev.append(nxt)
            nxt += 1
    for _ in range(tail):
        eu.append(nxt - 1), ev.append(nxt)
        nxt += 1
    perm = rng.permutation(nxt)
    eu, ev = perm[np.array(eu)], perm[np.array(ev)]
    extra = rng.integers(0, nxt, size=(2, nxt // 2))
    pairs = np.unique(np.stack([np.minimum(eu, ev), np.maximum(eu, ev)], 1), axis=0)
    more = np.unique(np.sort(extra[:, extra[0] != extra[1]], axis=0).T, axis=0) if hubs < 4 else pairs[:0]
    pairs = np.unique(np.concatenate([pairs, more]), axis=0)
    return _graph(nxt, pairs[:, 0], pairs[:, 1], rng.choice([1.0, 2.0, 3.5], size=len(pairs)), f"burst{hubs}x{leaves}")


@pytest.mark.parametrize("hubs,leaves,tail", [(1, 255, 0), (1, 256, 40), (2, 257, 1), (15, 273, 9), (16, 257, 300),
                                              (130, 270, 50), (70, 300, 5)])
def test_frontier_widths(B, hubs, leaves, tail):
    g = _burst(hubs, leaves, tail, np.random.default_rng(hubs * 1000 + leaves))
    for kind in (O.TREE_MAX_WEIGHT, O.TREE_FEGRASS):
        p = np.asarray(B.spanning_tree(g.n, g.row_ptr, g.col, g.w, kind=kind))
        assert np.array_equal(p, O.spanning_tree(g, kind)), (g.name, kind)


@pytest.mark.parametrize("size", [2, 3, 4, 5, 6, 8, 9, 36])
def test_forests_of_paths_between_empty_rows(B, size):
    """300 paths of `size` vertices, 45 isolated vertices after every third of them, equal weights throughout."""
    eu, ev, nxt = [], [], 40
    for k in range(300):
        for i in range(size - 1):
            eu.append(nxt + i), ev.append(nxt + i + 1)
        nxt += size + (45 if k % 3 == 0 else 0)
    g = _graph(nxt, np.array(eu), np.array(ev), np.ones(len(eu)), f"paths{size}")
    p = np.asarray(B.spanning_tree(g.n, g.row_ptr, g.col, g.w, kind=O.TREE_MAX_WEIGHT))
    assert np.array_equal(p, O.spanning_tree(g, O.TREE_MAX_WEIGHT))


def _without(g, drop):
    keep = np.ones(g.col.size, dtype=bool)
    keep[drop] = False
    rows = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    rp = np.zeros(g.n + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows[keep], minlength=g.n), out=rp[1:])
    return rp, np.ascontiguousarray(g.col[keep]), np.ascontiguousarray(g.w[keep])


@pytest.mark.parametrize("case", ["upper", "lower", "both", "weight_upper", "weight_lower", "last"])
def test_missing_mirror_images(B, case):
    g = W.grid_graph(30)
    rows = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    up, lo = np.flatnonzero(rows < g.col), np.flatnonzero(rows > g.col)
    rp, col, w = g.row_ptr, g.col, g.w.copy()
    if case == "upper":
        rp, col, w = _without(g, [up[700]])
    elif case == "lower":
        rp, col, w = _without(g, [lo[700]])
    elif case == "last":
        rp, col, w = _without(g, [g.col.size - 1])
    elif case == "both":  # as many above as below the diagonal, but not each other's images
        rp, col, w = _without(g, [up[3], lo[900]])
    else:
        w[(up if case == "weight_upper" else lo)[500]] *= 1.0 + 2.0**-52
    with pytest.raises(B.PdgError) as e:
        B.spanning_tree(g.n, rp, col, w, kind=O.TREE_MAX_WEIGHT)
    assert e.value.status == B.PDG_E_NOT_SYMMETRIC
    with pytest.raises(B.PdgError) as e:
        B.Sparsifier(g.n, rp, col, w, g.parent)
    assert e.value.status in (B.PDG_E_NOT_SYMMETRIC, B.PDG_E_NOT_A_TREE)  # a tree edge's entry may be the missing one
