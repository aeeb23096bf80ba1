"""Graphs whose weights come while the structure is worked on (host memory, at least 2^20 entries) and graphs read where
the caller keeps them (device memory): the same recovery as a small host graph takes, and the same refusals, weights
before the tree."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2508_20403_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2508_20403_gb300 import binding, build

    build.build()
    binding.load()
    return binding


@pytest.fixture(scope="module")
def mesh():
    g = W.mesh3d_graph(60, seed=4)
    assert g.col.size >= 1 << 20
    return g


def _arrays(g, where, **changed):
    import torch

    a = [np.array(changed.get(k, getattr(g, k))) for k in ("row_ptr", "col", "w", "parent")]
    if where == "host":
        return a
    t = [torch.from_numpy(x) for x in a]
    return [x.pin_memory() for x in t] if where == "pinned" else [x.cuda() for x in t]


def test_same_recovery(B, mesh):
    got = {}
    for where in ("host", "pinned", "device"):
        arrays = _arrays(mesh, where)
        with B.Sparsifier(mesh.n, *arrays) as sp:
            if where == "device":  # not read after the handle was made
                for x in arrays:
                    x.zero_()
            st, ids, sc, _ = sp.recover(0.05, 2)
            info = sp.info()
            got[where] = (st, np.array(ids), np.array(sc), info["m"], info["max_depth"])
    for where in ("pinned", "device"):
        for x, y in zip(got["host"], got[where]):
            assert np.array_equal(x, y), where


def _status(B, g, where, **changed):
    try:
        B.Sparsifier(g.n, *_arrays(g, where, **changed)).close()
        return B.PDG_OK
    except B.PdgError as e:
        return e.status


@pytest.mark.parametrize("where", ["host", "pinned", "device"])
def test_refusals(B, mesh, where):
    g = mesh
    row = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    lower = np.flatnonzero(row > g.col)

    def weight(at, x):
        w = g.w.copy()
        w[at] = x
        return w

    depth2 = next(v for v in range(g.n) if g.parent[v] >= 0 and g.parent[g.parent[v]] >= 0)
    cycle = g.parent.copy()
    cycle[g.parent[depth2]] = depth2
    stray = g.parent.copy()
    stray[int(np.flatnonzero(g.parent >= 0)[7])] = g.n - 1 if g.parent[7] != g.n - 1 else 0
    col = g.col.copy()
    col[[0, 1]] = col[[1, 0]]
    rows = g.row_ptr.copy()
    rows[500] = rows[501] + 1
    last = g.col.size - 1
    assert _status(B, g, where) == B.PDG_OK
    assert _status(B, g, where, w=weight(last, np.nan)) == B.PDG_E_BAD_WEIGHT
    assert _status(B, g, where, w=weight(lower[9000], g.w[lower[9000]] * (1 + 2.0**-52))) == B.PDG_E_NOT_SYMMETRIC
    assert _status(B, g, where, parent=cycle) == B.PDG_E_NOT_A_TREE
    assert _status(B, g, where, parent=stray) == B.PDG_E_NOT_A_TREE
    assert _status(B, g, where, parent=cycle, w=weight(5, -1.0)) == B.PDG_E_BAD_WEIGHT
    assert _status(B, g, where, parent=stray, w=weight(5, -1.0)) == B.PDG_E_BAD_WEIGHT
    assert _status(B, g, where, parent=cycle, w=weight(lower[3], 77.0)) == B.PDG_E_NOT_SYMMETRIC
    assert _status(B, g, where, col=col, w=weight(5, -1.0)) == B.PDG_E_NOT_CSR
    assert _status(B, g, where, row_ptr=rows, w=weight(5, -1.0)) == B.PDG_E_NOT_CSR
    tiny = g.w.copy()  # exponents further apart than the fixed-point range
    child = int(np.flatnonzero(g.parent >= 0)[11])
    for a, b in ((child, g.parent[child]), (g.parent[child], child)):
        p = g.row_ptr[a] + int(np.searchsorted(g.col[g.row_ptr[a]:g.row_ptr[a + 1]], b))
        tiny[p] = 2.0**-200
    assert _status(B, g, where, w=tiny) == B.PDG_E_RANGE
