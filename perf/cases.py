"""Performance cases of off-tree edge recovery: the calls a program makes through the public entry points.

Inputs are generated on the GPU (the workload families of paper_2508_20403_gb300.workloads: 2D grids, 3D 7-point
meshes, R-MAT, random geometric graphs, planar triangulations), from the seed alone, with the families' own weight
distributions.  Every graph gets its maximum-weight spanning tree from the library's own generator.

kind of a case
  recover  a resident handle (sparsify_init done once) that recovers again and again
  batch    a resident batch handle, one recover_offtree_batch for all its graphs
  serve    one request batch of the server: packed pinned host arrays -> sparsify_batch_init -> recover -> free
  oneshot  one graph end to end: sparsify_init -> recover -> endpoints of the recovered edges -> free
  tree     spanning-tree generation (either kind)
  pcg      the quality measure: a few preconditioned CG iterations with the recovered edges
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_20403_gb300 import binding as B

# ------------------------------------------------------------------------------------------------------- cases


def _case(name, kind, family, **kw):
    base = dict(kind=kind, family=family, sx=0, sy=0, sz=0, scale=0, n=0, graphs=1, alpha=0.05, c=2,
                score="stretch", replay=False, host=False, tree="max")
    assert set(kw) <= set(base), kw
    case = {**base, **kw}
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest ordinary call: a 100 x 100 grid kept resident, ids and scores to host arrays; launches and
        # round trips are what it costs
        _case("recover_grid100", "recover", "grid", sx=100, sy=100, alpha=0.02, host=True),
        # the headline workload: the 3D mesh resident, replayed from its CUDA graph, results left on the device
        _case("recover_mesh128", "recover", "mesh", sx=128, sy=128, sz=128, alpha=0.10, replay=True),
        # a ragged mesh with the paper's own score (resistance) and the widest neighbourhoods, launched plainly
        _case("recover_mesh_odd", "recover", "mesh", sx=97, sy=53, sz=71, alpha=0.05, c=3, score="resistance"),
        # the skewed social-graph shape at its largest size
        _case("recover_rmat22", "recover", "rmat", scale=22, alpha=0.02, replay=True),
        # a smaller skewed graph with a large budget: few, very uneven subtasks
        _case("recover_rmat17", "recover", "rmat", scale=17, alpha=0.10),
        # many graphs of uneven size in one launch (the batching mix), captured and replayed
        _case("batch_mix192", "batch", "mix", graphs=192, alpha=0.05, replay=True),
        # one request of the server on its own: a triangulation of 80,000 points from pinned host memory
        _case("serve_tri80k", "serve", "tri", n=80_000, alpha=0.05, host=True),
        # a server batch under load: a dozen graphs of the mix packed together
        _case("serve_mix12", "serve", "mix", graphs=12, alpha=0.10, host=True),
        # one mesh end to end from pinned host memory, endpoints of the recovered edges included
        _case("oneshot_mesh128", "oneshot", "mesh", sx=128, sy=128, sz=128, alpha=0.10, host=True),
        # the tree that recovery starts from, both kinds, graph on the device
        _case("tree_max_mesh128", "tree", "mesh", sx=128, sy=128, sz=128, tree="max"),
        _case("tree_fegrass_tri", "tree", "tri", n=300_000, tree="fegrass"),
        # how good the sparsifier is: the first preconditioned CG iterations on the grid with alpha*n edges
        _case("pcg_grid100", "pcg", "grid", sx=100, sy=100, alpha=0.05, host=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["recover", "recover", "recover", "batch", "serve", "oneshot", "tree", "pcg"])
    kw = dict(alpha=rng.choice([0.02, 0.05, 0.10]), c=rng.choice([1, 2, 2, 3]),
              score=rng.choice(["stretch", "stretch", "resistance"]), replay=rng.random() < 0.5,
              host=rng.random() < 0.5)
    if kind == "pcg":
        return _case("", kind, "grid", sx=rng.randint(30, 100), sy=rng.randint(30, 100), alpha=kw["alpha"], host=True)
    if kind == "batch":
        return _case("", kind, "mix", graphs=_log(rng, 3, 150), **kw)
    if kind == "serve":
        kw.update(replay=False, host=True)
        if rng.random() < 0.5:
            return _case("", kind, "tri", n=_log(rng, 10_000, 500_000), **kw)
        return _case("", kind, "mix", graphs=_log(rng, 1, 16), **kw)
    if kind == "oneshot":
        kw.update(replay=False)
    if kind == "tree":
        kw = dict(tree=rng.choice(["max", "fegrass"]))
    family = rng.choice(["grid", "mesh", "rmat", "tri", "rgg"])
    if family == "grid":
        return _case("", kind, family, sx=_log(rng, 30, 300), sy=_log(rng, 30, 300), **kw)
    if family == "mesh":
        return _case("", kind, family, sx=_log(rng, 12, 128), sy=_log(rng, 12, 128), sz=_log(rng, 12, 128), **kw)
    if family == "rmat":
        return _case("", kind, family, scale=rng.randint(11, 20), **kw)
    return _case("", kind, family, n=_log(rng, 1_000, 500_000), **kw)


# ---------------------------------------------------------------------------------------------- graph generation
# A graph is a dict of CUDA tensors: packed symmetric CSR (row_ptr, col, w), parent, and vtx_ptr (host int64).


def _pairs_grid(sx, sy):
    i = torch.arange(sx * sy, device="cuda").view(sx, sy)
    return (torch.cat([i[:, :-1].reshape(-1), i[:-1].reshape(-1)]), torch.cat([i[:, 1:].reshape(-1), i[1:].reshape(-1)]))


def _pairs_mesh(sx, sy, sz):
    i = torch.arange(sx * sy * sz, device="cuda").view(sx, sy, sz)
    a = torch.cat([i[:-1].reshape(-1), i[:, :-1].reshape(-1), i[:, :, :-1].reshape(-1)])
    b = torch.cat([i[1:].reshape(-1), i[:, 1:].reshape(-1), i[:, :, 1:].reshape(-1)])
    return a, b


def _pairs_rmat(shape, gen, scale, edge_factor=16):
    ne = edge_factor << scale
    u = torch.zeros(ne, dtype=torch.int64, device="cuda")
    v = torch.zeros_like(u)
    for lvl in range(scale):
        r = torch.rand(ne, generator=shape, device="cuda")
        u |= (r >= 0.76).long() << lvl
        v |= (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).long() << lvl
    perm = torch.randperm(1 << scale, generator=gen, device="cuda")
    return perm[u], perm[v]


def _pairs_tri(gen, n):
    """A planar triangulation of n randomly numbered points: square cells, each cut along a random diagonal."""
    sx = max(2, int(math.sqrt(n)))
    sy = max(2, n // sx)
    i = torch.arange(sx * sy, device="cuda").view(sx, sy)
    a, b = _pairs_grid(sx, sy)
    flip = torch.rand(sx - 1, sy - 1, generator=gen, device="cuda") < 0.5
    d0 = torch.where(flip, i[:-1, :-1], i[:-1, 1:]).reshape(-1)
    d1 = torch.where(flip, i[1:, 1:], i[1:, :-1]).reshape(-1)
    perm = torch.randperm(sx * sy, generator=gen, device="cuda")
    return sx * sy, perm[torch.cat([a, d0])], perm[torch.cat([b, d1])]


def _pairs_rgg(gen, sizes, degrees):
    """Random geometric graphs (one per entry of sizes) in unit squares, packed; points keep their random order."""
    sizes, degrees = np.asarray(sizes, dtype=np.int64), np.asarray(degrees, dtype=np.float64)
    radius = np.sqrt(degrees / (math.pi * sizes))
    side = np.maximum(1, np.floor(1.0 / radius)).astype(np.int64)
    base = np.concatenate([[0], np.cumsum(side * side)])
    dev = lambda x: torch.as_tensor(x, device="cuda")
    g = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), dev(sizes))
    N = int(sizes.sum())
    x = torch.rand(N, generator=gen, device="cuda", dtype=torch.float64)
    y = torch.rand(N, generator=gen, device="cuda", dtype=torch.float64)
    s = dev(side)[g]
    cx, cy = (x * s).long(), (y * s).long()
    cell, order = torch.sort(dev(base[:-1])[g] + cx * s + cy, stable=True)
    start = torch.zeros(int(base[-1]) + 1, dtype=torch.int64, device="cuda")
    start[1:] = torch.cumsum(torch.bincount(cell, minlength=int(base[-1])), 0)
    r2 = dev(radius * radius)[g]
    x, y, cx, cy, s, r2 = (t[order] for t in (x, y, cx, cy, s, r2))
    pos = torch.arange(N, device="cuda")
    us, vs = [], []
    for dx, dy in ((0, 0), (0, 1), (1, -1), (1, 0), (1, 1)):
        ok = (cx + dx < s) & (cy + dy < s) & (cy + dy >= 0)
        p = pos[ok]
        near = cell[p] + dx * s[p] + dy
        lo, hi = start[near], start[near + 1]
        if (dx, dy) == (0, 0):
            lo = p + 1
        cnt = hi - lo
        a = torch.repeat_interleave(p, cnt)
        first = torch.cumsum(cnt, 0) - cnt
        b = torch.arange(a.numel(), device="cuda") - torch.repeat_interleave(first - lo, cnt)
        keep = (x[a] - x[b]) ** 2 + (y[a] - y[b]) ** 2 <= r2[a]
        us.append(order[a[keep]])
        vs.append(order[b[keep]])
    return torch.cat(us), torch.cat(vs)


def _mix(gen, rng, graphs):
    """The batching mix: 70 % random geometric graphs, 30 % square grids, packed."""
    sizes, pa, pb, rsize, rdeg, rbase, at = [], [], [], [], [], [], 0
    for _ in range(graphs):
        if rng.random() < 0.7:
            n = int(round(math.exp(rng.uniform(math.log(1e3), math.log(2e5)))))
            rsize.append(n)
            rdeg.append(rng.uniform(6.0, 20.0))
            rbase.append(at)
        else:
            side = int(rng.integers(30, 301))
            n = side * side
            a, b = _pairs_grid(side, side)
            pa.append(a + at)
            pb.append(b + at)
        sizes.append(n)
        at += n
    if rsize:
        a, b = _pairs_rgg(gen, rsize, rdeg)
        # geometric graphs were numbered among themselves: move each to its own range
        own = np.concatenate([[0], np.cumsum(rsize)])[:-1]
        shift = torch.repeat_interleave(torch.as_tensor(np.asarray(rbase) - own, device="cuda"),
                                        torch.as_tensor(rsize, device="cuda"))
        pa.append(a + shift[a])
        pb.append(b + shift[b])
    return sizes, torch.cat(pa), torch.cat(pb)


def _csr(n, lo, hi, w):
    key, order = torch.sort(torch.cat([lo * n + hi, hi * n + lo]))
    row = key // n
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return row_ptr, (key % n).int(), torch.cat([w, w])[order]


def _roots(parent):
    r = torch.where(parent >= 0, parent.long(), torch.arange(parent.numel(), device="cuda"))
    while True:
        s = r[r]
        if torch.equal(s, r):
            return r
        r = s


def _graph(case, seed):
    # which vertices a random graph joins follows from the case (its sizes stay the same), how they are numbered
    # and what the edges weigh from the seed
    shape = torch.Generator(device="cuda").manual_seed(20250828 + case["scale"] + case["n"] + case["graphs"])
    rng = np.random.default_rng([20250828, case["n"], case["graphs"]])
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    fam = case["family"]
    if fam == "grid":
        sizes, (a, b) = [case["sx"] * case["sy"]], _pairs_grid(case["sx"], case["sy"])
    elif fam == "mesh":
        sizes, (a, b) = [case["sx"] * case["sy"] * case["sz"]], _pairs_mesh(case["sx"], case["sy"], case["sz"])
    elif fam == "rmat":
        sizes, (a, b) = [1 << case["scale"]], _pairs_rmat(shape, gen, case["scale"])
    elif fam == "tri":
        n, a, b = _pairs_tri(gen, case["n"])
        sizes = [n]
    elif fam == "rgg":
        sizes, (a, b) = [case["n"]], _pairs_rgg(shape, [case["n"]], [rng.uniform(6.0, 20.0)])
    else:
        sizes, a, b = _mix(shape, rng, case["graphs"])
    N = int(sum(sizes))
    key = torch.unique(torch.minimum(a, b) * N + torch.maximum(a, b))
    key = key[key // N != key % N]
    lo, hi = key // N, key % N
    u = torch.rand(key.numel(), generator=gen, device="cuda", dtype=torch.float64)
    if fam == "mesh":
        w = torch.pow(10.0, -3.0 + 6.0 * u)  # log-uniform over [1e-3, 1e3]
    elif fam == "rmat":
        w = 1.0 - u  # (0, 1]
    else:
        w = 1.0 + 9.0 * u  # [1, 10)
    vtx = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    row_ptr, col, wt = _csr(N, lo, hi, w)
    parent = torch.empty(N, dtype=torch.int32, device="cuda")
    B.spanning_tree(N, row_ptr, col, wt, kind=B.TREE_MAX_WEIGHT, parent_out=parent)
    if fam in ("rmat", "rgg", "mix"):  # keep the largest component of every graph
        root = _roots(parent)
        size = torch.bincount(root, minlength=N)
        g = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.as_tensor(sizes, device="cuda"))
        rank = size * (N + 1) + (N - torch.arange(N, device="cuda"))  # largest, then the smallest root
        best = torch.zeros(len(sizes), dtype=torch.int64, device="cuda").scatter_reduce(0, g, rank, "amax")
        keep = rank[root] == best[g]
        new = torch.cumsum(keep, 0) - 1
        ek = keep[lo]
        lo, hi, w = new[lo[ek]], new[hi[ek]], w[ek]
        p = parent[keep].long()
        parent = torch.where(p >= 0, new[p.clamp(min=0)], p).int()
        vtx = np.concatenate([[0], torch.cumsum(torch.bincount(g[keep], minlength=len(sizes)), 0).cpu().numpy()])
        N = int(vtx[-1])
        row_ptr, col, wt = _csr(N, lo, hi, w)
    return dict(n=N, row_ptr=row_ptr, col=col, w=wt, parent=parent, vtx_ptr=vtx.astype(np.int64))


class _HostGraph:
    """Host arrays of one graph, as the quality measure takes them."""

    def __init__(self, g):
        self.n = g["n"]
        self.row_ptr, self.col, self.w, self.parent = (g[k].cpu().numpy() for k in ("row_ptr", "col", "w", "parent"))


# ------------------------------------------------------------------------------------------------- prepare, run

PCG_ITERATIONS = 8  # rounding travels from one CG iteration to the next: the first ones are comparable


def _options(case):
    kw = dict(score_mode=B.SCORE_RESISTANCE if case["score"] == "resistance" else B.SCORE_STRETCH,
              use_graph=1 if case["replay"] else 0)
    if case["kind"] == "batch":  # the shape that the committed autotuner cache holds for large batches
        kw.update(block_tier_max=320, sort_tile_keys=4096)
    return B.default_options(**kw)


def _arrays(g, pinned):
    t = [g[k] for k in ("row_ptr", "col", "w", "parent")]
    return [x.cpu().pin_memory() for x in t] if pinned else t


def prepare(case, seed):
    g = _graph(case, seed)
    s = dict(case=case, n=g["n"], opt=_options(case))
    kind = case["kind"]
    alphas = np.full(len(g["vtx_ptr"]) - 1, case["alpha"])
    k = np.floor(alphas * np.diff(g["vtx_ptr"])).astype(np.int64)
    if kind == "recover":
        s["handle"] = B.Sparsifier(g["n"], *_arrays(g, False), options=s["opt"])
        if not case["host"]:
            s["ids"] = torch.zeros(max(int(k[0]), 1), dtype=torch.int32, device="cuda")
            s["scores"] = torch.zeros(max(int(k[0]), 1), dtype=torch.float64, device="cuda")
    elif kind == "batch":
        s["handle"] = B.BatchSparsifier(g["vtx_ptr"], *_arrays(g, False), options=s["opt"])
        s["alphas"] = alphas
        s["ids"] = torch.zeros(max(int(k.sum()), 1), dtype=torch.int32, device="cuda")
        s["scores"] = torch.zeros(max(int(k.sum()), 1), dtype=torch.float64, device="cuda")
    elif kind == "serve":
        s["alphas"], s["vtx_ptr"], s["arrays"] = alphas, g["vtx_ptr"], _arrays(g, True)
    elif kind == "oneshot":
        s["arrays"] = _arrays(g, case["host"])
        if not case["host"]:
            s["ids"] = torch.zeros(max(int(k[0]), 1), dtype=torch.int32, device="cuda")
            s["scores"] = torch.zeros(max(int(k[0]), 1), dtype=torch.float64, device="cuda")
    elif kind == "tree":
        s["arrays"] = _arrays(g, False)[:3]
        s["parent"] = torch.empty(g["n"], dtype=torch.int32, device="cuda")
    else:
        s["graph"] = _HostGraph(g)
        s["b"] = np.random.default_rng([int(seed), 5]).standard_normal(g["n"])
        with B.Sparsifier(g["n"], *_arrays(g, False)) as sp:
            s["edges"] = np.array(sp.recover(case["alpha"], case["c"])[1])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "recover":
        st, ids, scores, _ = s["handle"].recover(case["alpha"], case["c"], s.get("ids"), s.get("scores"))
        return dict(status=st, ids=ids, scores=scores)
    if kind == "batch":
        _, _, ids, scores, counts, status = s["handle"].recover_batch(s["alphas"], case["c"], None, s["ids"], s["scores"])
        return dict(ids=ids, scores=scores, counts=counts, status=status)
    if kind == "serve":
        with B.BatchSparsifier(s["vtx_ptr"], *s["arrays"], options=s["opt"]) as bs:
            _, _, ids, scores, counts, status = bs.recover_batch(s["alphas"], case["c"])
        return dict(ids=ids, scores=scores, counts=counts, status=status)
    if kind == "oneshot":
        with B.Sparsifier(s["n"], *s["arrays"], options=s["opt"]) as sp:
            st, ids, scores, _ = sp.recover(case["alpha"], case["c"], s.get("ids"), s.get("scores"))
            u, v = sp.endpoints(ids)
        return dict(status=st, ids=ids, scores=scores, u=u, v=v)
    if kind == "tree":
        tree = B.TREE_FEGRASS if case["tree"] == "fegrass" else B.TREE_MAX_WEIGHT
        return dict(parent=B.spanning_tree(s["n"], *s["arrays"], kind=tree, parent_out=s["parent"]))
    it, rel, history, z = B.pcg_trace(s["graph"], s["edges"], s["b"], tol=1e-3, max_iter=PCG_ITERATIONS)
    return dict(iterations=it, residual=rel, history=history, preconditioned=z)


# -------------------------------------------------------------------------------------------------------- work


def _sizes(case):
    """(vertices, edges) of a case, the expected ones where the graph is random."""
    fam = case["family"]
    if fam == "grid":
        sx, sy = case["sx"], case["sy"]
        return sx * sy, 2 * sx * sy - sx - sy
    if fam == "mesh":
        sx, sy, sz = case["sx"], case["sy"], case["sz"]
        return sx * sy * sz, 3 * sx * sy * sz - sx * sy - sx * sz - sy * sz
    if fam == "rmat":
        return 0.57 * 2.0 ** case["scale"], 15.3 * 2.0 ** case["scale"]
    if fam == "tri":
        return case["n"], 3.0 * case["n"]
    if fam == "rgg":
        return case["n"], 6.5 * case["n"]
    mean = 0.7 * (2e5 - 1e3) / math.log(200.0) + 0.3 * (300.0 ** 3 - 30.0 ** 3) / (3 * 270.0)
    edges = 0.7 * 6.5 * (2e5 - 1e3) / math.log(200.0) + 0.6 * (300.0 ** 3 - 30.0 ** 3) / (3 * 270.0)
    return case["graphs"] * mean, case["graphs"] * edges


def work(case):
    n, m = _sizes(case)
    k = case["alpha"] * n
    kind = case["kind"]
    csr = 8.0 * (n + 1) + 24.0 * m
    if kind in ("recover", "batch"):  # the resident edges (two ends, weight) and tree in, ids and scores out
        return dict(bytes=16.0 * m + 4.0 * n + 12.0 * k, flops=0.0)
    if kind == "serve":
        return dict(bytes=csr + 4.0 * n + 12.0 * k, flops=0.0)
    if kind == "oneshot":
        return dict(bytes=csr + 4.0 * n + 20.0 * k, flops=0.0)
    if kind == "tree":
        return dict(bytes=csr + 4.0 * n, flops=0.0)
    # per iteration: the k x k solve and one product with the Laplacian; once: factorising the k x k matrix
    return dict(bytes=csr + 4.0 * n + 16.0 * n + 4.0 * k,
                flops=2.0 * k ** 3 / 3.0 + (PCG_ITERATIONS + 1) * (2.0 * k * k + 4.0 * m + 10.0 * n))


# ------------------------------------------------------------------------------------------------------- exact


def _tree_numbers(parent, wup):
    """Depth and root distance (sum of 1/w) of every vertex, and the binary-lifting ancestor table."""
    n = parent.numel()
    up = torch.where(parent >= 0, parent.long(), torch.arange(n, device=parent.device))
    depth = (parent >= 0).long()
    dist = torch.where(parent >= 0, 1.0 / wup, torch.zeros_like(wup))
    table, at = [up], up
    while True:
        depth, dist, nxt = depth + depth[at], dist + dist[at], at[at]
        if torch.equal(nxt, at):
            return depth, dist, table
        at = nxt
        table.append(at)


def _lca(u, v, depth, table):
    u, v = torch.where(depth[u] >= depth[v], u, v), torch.where(depth[u] >= depth[v], v, u)
    gap = depth[u] - depth[v]
    for j, t in enumerate(table):
        u = torch.where((gap >> j) & 1 == 1, t[u], u)
    for t in reversed(table):
        differ = t[u] != t[v]
        u, v = torch.where(differ, t[u], u), torch.where(differ, t[v], v)
    return torch.where(u == v, u, table[0][u])


def _greedy(order, u, v, lca, hops_u, hops_v, parent, c, k):
    """The first k recovered edges of `order`, or all survivors: an edge is skipped when an earlier recovered edge
    of its LCA has both its ends within that edge's neighbourhoods (either way round)."""
    def up(x):
        chain = [x]
        while len(chain) <= c and chain[-1] >= 0:
            chain.append(parent[chain[-1]])
        return [y for y in chain if y >= 0]

    marks, got = {}, []
    for e in order:
        l, cu, cv = lca[e], up(u[e]), up(v[e])
        hit = False
        for a, b in ((cu, cv), (cv, cu)):
            for i, x in enumerate(a):
                for j, y in enumerate(b):
                    for si, sj in marks.get((l, x, y), ()):
                        hit = hit or (si >= i and sj >= j)
        if hit:
            continue
        got.append(e)
        if len(got) == k:
            break
        beta = min(hops_u[e], hops_v[e], c)
        for i in range(beta + 1):
            for j in range(beta + 1):
                marks.setdefault((l, cu[i], cv[j]), []).append((beta - i, beta - j))
    return got


EXACT_EDGES = 20_000  # the sequential walk of more edges takes too long


def _exact_scores(g, lo, hi, alpha, c, score):
    """Scores of the recovered edges of one graph (vertices lo .. hi of the packed arrays), in recovery order."""
    rp, n = g["row_ptr"][lo:hi + 1], hi - lo
    e0, e1 = int(rp[0]), int(rp[-1])
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    col, w = g["col"][e0:e1].long() - lo, g["w"][e0:e1]
    parent = g["parent"][lo:hi].long()
    parent = torch.where(parent >= 0, parent - lo, parent)
    wup = torch.ones(n, dtype=torch.float64, device="cuda")
    tree = parent[row] == col
    wup[row[tree]] = w[tree]
    off = (row < col) & (parent[row] != col) & (parent[col] != row)
    u, v, w = row[off], col[off], w[off]
    depth, dist, table = _tree_numbers(parent, wup)
    l = _lca(u, v, depth, table)
    s = dist[u] + dist[v] - 2.0 * dist[l]
    if score == "stretch":
        s = s * w
    k = int(math.floor(alpha * n))
    order = torch.sort(s, descending=True, stable=True)[1].cpu().tolist()
    host = [t.cpu().tolist() for t in (u, v, l, depth[u] - depth[l], depth[v] - depth[l], parent)]
    got = _greedy(order, *host, c, k) if k > 0 else []
    return s.cpu().numpy()[np.asarray(got, dtype=np.int64)]


def _exact_pcg(case, seed):
    """The same iteration with a dense Cholesky factor of the grounded sparsifier Laplacian."""
    s = prepare(case, seed)
    g, n = s["graph"], s["n"]
    t = lambda x: torch.as_tensor(x, device="cuda")
    rp, col, w, parent, ids, b = t(g.row_ptr), t(g.col).long(), t(g.w), t(g.parent).long(), t(s["edges"]).long(), t(s["b"])
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    upper = row < col
    eu, ev, ew = row[upper], col[upper], w[upper]
    keep = (parent[eu] == ev) | (parent[ev] == eu)
    keep[ids] = True
    P = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    pu, pv, pw = eu[keep], ev[keep], ew[keep]
    for a, c, x in ((pu, pv, -pw), (pv, pu, -pw), (pu, pu, pw), (pv, pv, pw)):
        P.index_put_((a, c), x, accumulate=True)
    free = parent >= 0
    L = torch.linalg.cholesky(P[free][:, free])

    def solve(r):
        z = torch.zeros_like(r)
        z[free] = torch.cholesky_solve(r[free, None], L)[:, 0]
        return z - z.mean()

    def product(x):
        y = torch.zeros_like(x)
        d = ew * (x[eu] - x[ev])
        return y.index_add_(0, eu, d).index_add_(0, ev, -d)

    r = b - b.mean()
    norm = r.norm()
    z = first = solve(r)
    p, rz, history = z.clone(), r @ z, []
    for _ in range(PCG_ITERATIONS):
        q = product(p)
        a = rz / (p @ q)
        r = r - a * q
        history.append(float(r.norm() / norm))
        if history[-1] <= 1e-3:
            break
        z = solve(r)
        rz, old = r @ z, rz
        p = z + (rz / old) * p
    return dict(iterations=None, residual=history[-1], history=np.asarray(history), preconditioned=first.cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "tree":  # whole numbers only
        return None
    if kind == "pcg":
        return _exact_pcg(case, seed)
    if case["alpha"] * _sizes(case)[0] > EXACT_EDGES:
        return None
    g = _graph(case, seed)
    vtx = [int(x) for x in g["vtx_ptr"]]
    parts = [_exact_scores(g, a, b, case["alpha"], case["c"], case["score"]) for a, b in zip(vtx, vtx[1:])]
    out = dict(ids=None, status=None)
    if kind in ("recover", "oneshot"):
        out["scores"] = parts[0]
        if kind == "oneshot":
            out.update(u=None, v=None)
        return out
    # packed results: graph g's scores start at its budget's offset, unused places are zero or left alone
    if any(len(p) != int(math.floor(case["alpha"] * (b - a))) for p, a, b in zip(parts, vtx, vtx[1:])):
        return None
    out.update(scores=np.concatenate(parts), counts=None)
    return out
