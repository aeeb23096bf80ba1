"""An entry without an equal mirror image is refused as asymmetry by every init, whatever else is wrong with the graph for
want of it (a tree edge that is not there any more): device arrays, host arrays, and host arrays whose weights come
late."""
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


def _without(g, drop):
    keep = np.ones(g.col.size, dtype=bool)
    keep[drop] = False
    rows = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    rp = np.zeros(g.n + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows[keep], minlength=g.n), out=rp[1:])
    return rp, np.ascontiguousarray(g.col[keep]), np.ascontiguousarray(g.w[keep])


def _entry(g, u, v):
    return int(g.row_ptr[u] + np.searchsorted(g.col[g.row_ptr[u]:g.row_ptr[u + 1]], v))


@pytest.mark.parametrize("edge", ["tree", "off"])
@pytest.mark.parametrize("case", ["upper", "lower", "both", "weight_upper", "weight_lower"])
@pytest.mark.parametrize("graph", ["grid", "mesh"])
def test_missing_mirror_images(B, graph, case, edge):
    g = W.grid_graph(30) if graph == "grid" else W.mesh3d_graph(60)  # the mesh has more than 2^20 entries
    rows = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
    tree = (g.parent[rows] == g.col) | (g.parent[g.col] == rows)
    of_kind = tree if edge == "tree" else ~tree
    up, lo = np.flatnonzero((rows < g.col) & of_kind), np.flatnonzero((rows > g.col) & of_kind)
    rp, col, w = g.row_ptr, g.col, g.w.copy()
    if case == "upper":
        rp, col, w = _without(g, [up[200]])
    elif case == "lower":
        rp, col, w = _without(g, [lo[200]])
    elif case == "both":  # as many above as below the diagonal, but not each other's images
        assert _entry(g, int(g.col[up[3]]), int(rows[up[3]])) != lo[300]
        rp, col, w = _without(g, [up[3], lo[300]])
    else:
        w[(up if case == "weight_upper" else lo)[150]] *= 1.0 + 2.0**-52
    import torch

    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt).cuda()
    host = (rp, col, w, g.parent)
    device = (t(rp, torch.int64), t(col, torch.int32), t(w, torch.float64), t(g.parent, torch.int32))
    for arrays in (host, device):
        with pytest.raises(B.PdgError) as e:
            B.Sparsifier(g.n, *arrays)
        assert e.value.status == B.PDG_E_NOT_SYMMETRIC
