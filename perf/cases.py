"""The workloads this library is timed on: its public entry points over the sizes, graph families, block
widths and storage types that the repository's configurations, tests and benchmark use.

A graph case names a family and its sizes, which fix its edges; the seed draws the weights, the order of the
edge list where it has none of its own, and the random vectors, all on the GPU:
  grid2d   a x b 4-neighbour grid, weights U[1, 10)
  grid3d   s^3 6-neighbour grid, weights 10^U[-2, 2)
  thermal  nx x ny x nz layered 6-neighbour mesh, one conductivity 10^U[-1, 2) per layer
  power    side^2 grid plus 1% via edges within distance 8, weights LogNormal(0, 1.5)
  chung_lu power-law graph, mean degree 16, exponent 2.3, weights U[0.5, 2), edges in random order
  knn      10-nearest-neighbour graphs of uniform points in the unit cube, points in random order
"""
import math

import numpy as np
import torch

import paper_2008_07633_gb300.sfg as S

DEV = "cuda:0"
BF16, F32 = "bf16", "f32"
NFEAT, HID = 16, 64


def listed():
    return [
        # The smallest call: the paper-sized 64 x 64 grid through the whole flat method (Algorithm 1). Launches and waits count.
        {"name": "sparsify_grid2d_64", "kind": "sparsify", "family": "grid2d", "a": 64, "b": 64, "K": 8, "steps": 10, "levels": 0,
         "budget": 0.1, "unit": 1, "mode": 0, "storage": F32},
        # A small layered thermal mesh, filtered, scored and selected: one step of an interactive loop over small graphs.
        {"name": "filter_thermal_17k", "kind": "filter", "family": "thermal", "nx": 40, "ny": 36, "nz": 12, "K": 16, "steps": 15,
         "budget": 0.05, "mode": 0, "storage": F32},
        # The benchmark's headline step: filter + score + selection on the 128^3 grid, FP32 blocks of 32 vectors.
        {"name": "filter_grid3d_128", "kind": "filter", "family": "grid3d", "s": 128, "K": 32, "steps": 20,
         "budget": 0.05, "mode": 0, "storage": F32},
        # The precision configuration: a 2048^2 power grid with BF16 blocks of 64 vectors.
        {"name": "filter_power_2048_bf16", "kind": "filter", "family": "power", "side": 2048, "K": 64, "steps": 20,
         "budget": 0.05, "mode": 0, "storage": BF16},
        # A power-law graph with hub rows: the gathers are random and most of them miss the cache.
        {"name": "filter_chung_lu_1m", "kind": "filter", "family": "chung_lu", "n": 1 << 20, "K": 32, "steps": 20,
         "budget": 0.05, "mode": 0, "storage": F32},
        # The plain method of the paper: two-level coarsening, backward mapping and edge recovery, hierarchy returned.
        {"name": "sparsify_2level_grid3d_128", "kind": "sparsify", "family": "grid3d", "s": 128, "K": 32, "steps": 20, "levels": 2,
         "budget": 0.05, "unit": 0, "mode": 0, "storage": F32},
        # A new graph arriving as an unordered edge list: canonical form and CSR Laplacian of 8M power-law edges.
        {"name": "laplacian_chung_lu_1m", "kind": "laplacian", "family": "chung_lu", "n": 1 << 20},
        # Many graphs of uneven size through one batch plan (the plan is kept, each seed is a run).
        {"name": "batch_knn_64", "kind": "batch", "ng": 64, "lo": 1000, "hi": 100000, "K": 16, "steps": 15, "budget": 0.05,
         "mode": 0, "storage": F32},
        # Learned proposals: the network over every off-tree edge of a large graph; a row count that fills no last tile.
        {"name": "mlp_forward_8m", "kind": "mlp_forward", "rows": 8000003},
        # Learned proposals: the gradient of one training batch (65,536 rows is the default batch).
        {"name": "mlp_gradient_64k", "kind": "mlp_gradient", "rows": 65536},
        # The paper's own relaxation: two Gauss-Seidel sweeps in colour order on a 1M-node mesh.
        {"name": "smooth_gs_thermal_1m", "kind": "smooth_gs", "family": "thermal", "nx": 128, "ny": 128, "nz": 64, "K": 32, "steps": 2,
         "storage": F32},
        # End to end on a new graph: edge list to Laplacian to flat sparsifier on the 128^3 grid.
        {"name": "end_to_end_grid3d_128", "kind": "end_to_end", "family": "grid3d", "s": 128, "K": 32, "steps": 20, "levels": 0,
         "budget": 0.05, "unit": 0, "mode": 0, "storage": F32},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_family(rng, top, families):
    """A family and its sizes, about n nodes with n log-uniform in [1000, top]."""
    fam = rng.choice(families)
    n = _log_int(rng, 1000, top)
    if fam == "grid2d":
        a = max(2, int(round(math.sqrt(n) * rng.uniform(0.3, 1.7))))
        return {"family": fam, "a": a, "b": max(2, n // a)}
    if fam == "grid3d":
        return {"family": fam, "s": max(10, int(round(n ** (1 / 3))))}
    if fam == "thermal":
        nz = rng.randint(3, max(4, int(round(n ** (1 / 3)))))
        nx = max(3, int(round(math.sqrt(n / nz) * rng.uniform(0.5, 1.5))))
        return {"family": fam, "nx": nx, "ny": max(3, n // (nz * nx)), "nz": nz}
    if fam == "power":
        return {"family": fam, "side": max(24, int(round(math.sqrt(n))))}
    return {"family": fam, "n": max(1000, n // 4)}  # chung_lu: eight times the edges of a mesh


def draw(rng):
    meshes = ["grid2d", "grid3d", "thermal", "power"]
    kind = rng.choice(["filter"] * 4 + ["sparsify"] * 2 + ["laplacian", "batch", "mlp_forward", "mlp_gradient", "smooth_gs", "end_to_end"])
    if kind == "mlp_forward":
        return {"kind": kind, "rows": _log_int(rng, 500, 8000000)}
    if kind == "mlp_gradient":
        return {"kind": kind, "rows": _log_int(rng, 500, 4000000)}
    if kind == "laplacian":
        return {"kind": kind, **_draw_family(rng, 4000000, meshes + ["chung_lu"])}
    storage = rng.choice([F32, F32, BF16])
    K = rng.choice([8, 16, 32, 64] if storage == BF16 else [4, 8, 16, 32, 64])
    c = {"kind": kind, "K": K, "steps": rng.randint(5, 20), "storage": storage}
    if kind == "smooth_gs":
        return {**c, "steps": rng.randint(1, 4), **_draw_family(rng, min(1000000, 32000000 // K), meshes)}
    c["mode"] = rng.choice([0, 0, 1, 2])
    c["budget"] = rng.choice([0.01, 0.05, 0.1])
    if kind == "batch":
        lo = _log_int(rng, 1000, 4000)
        return {**c, "K": min(K, 32), "ng": rng.randint(3, 64), "lo": lo, "hi": lo * rng.randint(2, 20)}
    top = min(2000000, 64000000 // K)
    if kind == "filter":
        return {**c, **_draw_family(rng, top, meshes + ["chung_lu"])}
    c.update(unit=rng.choice([0, 1]), levels=rng.randint(0, 2) if kind == "sparsify" else 0)
    return {**c, **_draw_family(rng, top // (2 if c["levels"] else 1), meshes + ["chung_lu"])}


# ------------------------------------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed & 0x7FFFFFFF)


def _uniform(g, m, lo, hi):
    return torch.rand(m, generator=g, device=DEV) * (hi - lo) + lo


def _mesh(shape):
    """Endpoints along every axis of a row-major lattice, one (u, v) pair of flat tensors per axis, last axis first."""
    idx = torch.arange(math.prod(shape), dtype=torch.int32, device=DEV).reshape(shape)
    out = []
    for d in reversed(range(len(shape))):
        k = shape[d]
        out.append((idx.narrow(d, 0, k - 1).reshape(-1), idx.narrow(d, 1, k - 1).reshape(-1)))
    return out


def _shape():
    """The generator of a case's own edges: the same for every seed."""
    return _gen(1234)


def _knn(n, shape, g, k=10, room=16):
    """About the 10 nearest neighbours of n uniform points: the nearest among the points of the 27 cells around each point's
    cell (4 points a cell on average, up to 16 looked at). Repeated pairs are left to the Laplacian."""
    pts = torch.rand((n, 3), generator=shape, device=DEV)
    c = max(1, int((n / 4) ** (1 / 3)))
    cell = (pts * c).long().clamp_(0, c - 1)
    cid = (cell[:, 0] * c + cell[:, 1]) * c + cell[:, 2]
    order = torch.argsort(cid, stable=True)
    count = torch.bincount(cid, minlength=c ** 3)
    start = torch.cumsum(count, 0) - count
    place = torch.arange(n, device=DEV) - start[cid[order]]
    table = torch.full((c ** 3, room), -1, dtype=torch.long, device=DEV)
    keep = place < room
    table[cid[order][keep], place[keep]] = order[keep]
    near = torch.arange(-1, 2, device=DEV)
    offs = torch.cartesian_prod(near, near, near)
    nb = cell[:, None, :] + offs[None]
    inside = ((nb >= 0) & (nb < c)).all(2)
    nb = nb.clamp(0, c - 1)
    cand = table[(nb[..., 0] * c + nb[..., 1]) * c + nb[..., 2]]
    cand = torch.where(inside[..., None], cand, -1).reshape(n, -1)
    me = torch.arange(n, device=DEV)[:, None]
    d2 = ((pts[cand.clamp_min(0)] - pts[:, None, :]) ** 2).sum(2)
    d2 = torch.where((cand < 0) | (cand == me), float("inf"), d2)
    best, at = torch.topk(d2, k, dim=1, largest=False)
    j = cand.gather(1, at)
    ok = torch.isfinite(best).reshape(-1)
    u, v, d2 = me.expand(n, k).reshape(-1)[ok], j.reshape(-1)[ok], best.reshape(-1)[ok]
    first = (u < v) | ~(j[v] == u[:, None]).any(1)  # a pair that both ends list is kept once
    u, v, d2 = u[first], v[first], d2[first]
    w = torch.exp(-d2 / d2.sqrt().mean() ** 2).clamp_min(1e-30) * _uniform(g, u.numel(), 0.9, 1.1)
    return n, u.int(), v.int(), w.float()


def _edges(case, seed):
    """(n, u, v, w) of the case's graph on the device."""
    g, fam = _gen(seed), case["family"]
    if fam in ("grid2d", "grid3d"):
        shape = (case["a"], case["b"]) if fam == "grid2d" else (case["s"],) * 3
        axes = _mesh(shape)
        u, v = torch.cat([a[0] for a in axes]), torch.cat([a[1] for a in axes])
        w = _uniform(g, u.numel(), 1.0, 10.0) if fam == "grid2d" else torch.pow(10.0, _uniform(g, u.numel(), -2.0, 2.0))
        return math.prod(shape), u, v, w
    if fam == "thermal":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        k = torch.pow(10.0, _uniform(g, nz, -1.0, 2.0))
        axes = _mesh((nz, ny, nx))
        kz = 2 * k[:-1] * k[1:] / (k[:-1] + k[1:])
        w = torch.cat([k.repeat_interleave(ny * (nx - 1)), k.repeat_interleave((ny - 1) * nx), kz.repeat_interleave(ny * nx)])
        u, v = torch.cat([a[0] for a in axes]), torch.cat([a[1] for a in axes])
        return nx * ny * nz, u, v, w * _uniform(g, w.numel(), 0.9, 1.1)
    if fam == "power":
        side, r = case["side"], 8
        n = side * side
        axes = _mesh((side, side))
        offs = torch.tensor([(x, y) for x in range(-r, r + 1) for y in range(-r, r + 1) if 0 < x * x + y * y <= r * r and abs(x) + abs(y) > 1],
                            dtype=torch.int32, device=DEV)
        nv = int(0.01 * n)
        shape = _shape()
        p = torch.randint(0, n, (nv,), generator=shape, device=DEV, dtype=torch.int32)
        o = offs[torch.randint(0, offs.shape[0], (nv,), generator=shape, device=DEV)]
        i, j = p // side + o[:, 0], p % side + o[:, 1]
        ok = (i >= 0) & (i < side) & (j >= 0) & (j < side)
        u, v = torch.cat([a[0] for a in axes] + [p[ok]]), torch.cat([a[1] for a in axes] + [(i * side + j)[ok]])
        return n, u, v, torch.exp(1.5 * torch.randn(u.numel(), generator=g, device=DEV))
    n, gamma, deg = case["n"], 2.3, 16.0  # chung_lu
    theta = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) ** (-1.0 / (gamma - 1.0))
    theta = theta * (deg * n / theta.sum())
    theta = torch.minimum(theta, theta.sum().sqrt())
    cdf = torch.cumsum(theta, 0)
    cdf = cdf / cdf[-1].clone()
    pairs = int(n * deg / 2)
    shape = _shape()
    u = torch.searchsorted(cdf, torch.rand(pairs, generator=shape, device=DEV, dtype=torch.float64)).clamp_max_(n - 1)
    v = torch.searchsorted(cdf, torch.rand(pairs, generator=shape, device=DEV, dtype=torch.float64)).clamp_max_(n - 1)
    order = torch.randperm(pairs, generator=g, device=DEV)
    return n, u[order].int(), v[order].int(), _uniform(g, pairs, 0.5, 2.0)


def _theta(g):
    """Network parameters of the size training gives: Kaiming-uniform weights, small biases."""
    def kaiming(fan, *shape):
        return (torch.rand(shape, generator=g, device=DEV) * 2 - 1) * math.sqrt(6 / fan)
    parts = [kaiming(NFEAT, NFEAT, HID), 0.1 * torch.randn(HID, generator=g, device=DEV), kaiming(HID, HID, HID),
             0.1 * torch.randn(HID, generator=g, device=DEV), kaiming(HID, HID), 0.1 * torch.randn(1, generator=g, device=DEV)]
    return torch.cat([p.reshape(-1) for p in parts])


def _features(g, rows):
    """Rows shaped like an edge's features: logarithms of weights, degrees and distances in the first eight columns, zeros after."""
    mean = torch.tensor([0.0, 4.0, 0.8, -1.0, 0.5, 1.5, 5.0, 0.7], device=DEV)
    x = torch.zeros((rows, NFEAT), device=DEV)
    x[:, :8] = torch.randn((rows, 8), generator=g, device=DEV) + mean
    x[:, 2].abs_()
    return x


def _mlp_inputs(case, seed):
    g = _gen(seed)
    theta, x = _theta(g), _features(g, case["rows"])
    return theta, x, 2.0 * torch.randn(case["rows"], generator=g, device=DEV) - 2.0


def _batch_sizes(case):
    u = np.random.default_rng(3).uniform(math.log(case["lo"]), math.log(case["hi"]), case["ng"])
    return [int(x) for x in np.rint(np.exp(u))]


def _storage(case):
    return torch.bfloat16 if case["storage"] == BF16 else torch.float32


def _filter_k(case, n, candidates):
    return min(candidates, int(case["budget"] * n + 0.5))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed, "ctx": S.sfg_ctx_create(0)}
    ctx = st["ctx"]
    if kind in ("mlp_forward", "mlp_gradient"):
        theta, st["x"], st["t"] = _mlp_inputs(case, seed)
        st["net"] = S.sfg_mlp_create(ctx, seed)
        S.sfg_mlp_set_params(ctx, st["net"], theta)
        return st
    if kind == "batch":
        shape, g = _shape(), _gen(seed)
        graphs = [S.sfg_laplacian(ctx, *_knn(n, shape, g)) for n in _batch_sizes(case)]
        st["plan"] = S.Batch(ctx, graphs, K=case["K"], steps=case["steps"], mode=case["mode"], budget_frac=case["budget"],
                             storage=_storage(case))
        return st
    n, u, v, w = _edges(case, seed)
    if kind in ("laplacian", "end_to_end"):  # these start from the edge list
        st["edges"] = (n, u, v, w)
        return st
    st["g"] = S.sfg_laplacian(ctx, n, u, v, w)
    if kind == "filter":  # the sparsifier so far: the maximum spanning forest; candidates: every edge outside it
        mask, _ = S.sfg_spanning_tree(ctx, st["g"])
        st["p"] = S.sfg_graph_subgraph(ctx, st["g"], mask)
        st["ids"] = torch.nonzero(mask == 0).reshape(-1).int()
        st["k"] = _filter_k(case, n, st["ids"].numel())
    if kind == "smooth_gs":  # the colouring stays with the graph
        S.sfg_coloring(ctx, st["g"])
    return st


def _sparsify(ctx, g, case, seed, **more):
    return S.sfg_sparsify(ctx, g, K=case["K"], steps=case["steps"], levels=case["levels"], seed=seed, mode=case["mode"],
                          budget_frac=case["budget"], budget_unit=case["unit"], storage=_storage(case), **more)


def run(st):
    case, ctx, seed, kind = st["case"], st["ctx"], st["seed"], st["case"]["kind"]
    if kind == "filter":
        scores = S.sfg_filter_score(ctx, st["g"], st["p"], st["ids"], case["K"], case["steps"], seed=seed, storage=_storage(case),
                                    mode=case["mode"])
        return {"scores": scores, "selected": S.sfg_select_topk(ctx, scores, st["ids"], st["k"])}
    if kind == "sparsify":
        if not case["levels"]:
            mask, count = _sparsify(ctx, st["g"], case, seed)
            return {"mask": mask, "count": count}
        mask, count, h = _sparsify(ctx, st["g"], case, seed, hierarchy=True)
        agg, f2c = h.map(1)
        return {"mask": mask, "count": count, "agg": agg, "f2c": f2c}
    if kind == "end_to_end":
        g = S.sfg_laplacian(ctx, *st["edges"])
        mask, count = _sparsify(ctx, g, case, seed)
        u, v, w = S.sfg_graph_edges(ctx, g)
        return {"u": u, "v": v, "w": w, "mask": mask, "count": count}
    if kind == "laplacian":
        g = S.sfg_laplacian(ctx, *st["edges"])
        row_ptr, col, val, eid, deg = S.sfg_graph_csr(ctx, g)
        return {"row_ptr": row_ptr, "col": col, "val": val, "eid": eid, "deg": deg}
    if kind == "batch":
        return {"mask": st["plan"].run(seed)}
    if kind == "mlp_forward":
        return {"y": S.sfg_mlp_forward(ctx, st["net"], st["x"])}
    if kind == "mlp_gradient":
        grad, loss = S.sfg_mlp_gradient(ctx, st["net"], st["x"], st["t"])
        return {"grad": grad, "loss": loss}
    return {"x": S.sfg_smooth_gs(ctx, st["g"], case["K"], case["steps"], seed=seed, storage=_storage(case))}


# ------------------------------------------------------------------------------------------------ work

def _size(case):
    """Nodes and edges (power-law and k-NN graphs: about)."""
    f = case.get("family")
    if f == "grid2d":
        a, b = case["a"], case["b"]
        return a * b, 2 * a * b - a - b
    if f == "grid3d":
        s = case["s"]
        return s ** 3, 3 * s * s * (s - 1)
    if f == "thermal":
        x, y, z = case["nx"], case["ny"], case["nz"]
        return x * y * z, 3 * x * y * z - x * y - y * z - x * z
    if f == "power":
        s = case["side"]
        return s * s, 2 * s * (s - 1) + int(0.01 * s * s)
    if f == "chung_lu":
        return case["n"], int(7.5 * case["n"])
    n = int(case["ng"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"]))
    return n, int(5.8 * n)


def work(case):
    """Each input read once, each output written once; multiply-adds of the sweeps, scores and matrix products count two."""
    kind = case["kind"]
    if kind == "mlp_forward":
        return {"bytes": case["rows"] * (4 * NFEAT + 4) + 4 * 5313, "flops": case["rows"] * 2 * (NFEAT * HID + HID * HID + HID)}
    if kind == "mlp_gradient":  # forward, the same again for the weights, and the second layer's backward
        per_row = 2 * (2 * (NFEAT * HID + HID * HID + HID) + HID * HID + HID)
        return {"bytes": case["rows"] * (4 * NFEAT + 4) + 2 * 4 * 5313, "flops": case["rows"] * per_row}
    n, m = _size(case)
    edges, csr = 12 * m, 24 * m + 12 * n  # (u, v, w); (column, weight, edge id) per entry, row bounds and degree per node
    if kind == "laplacian":
        return {"bytes": edges + csr, "flops": 2 * m}
    K, T = case["K"], case["steps"]
    block = n * K * (2 if case["storage"] == BF16 else 4)
    sweep_g, sweep_p = 2 * K * (2 * m + n), 2 * K * 3 * n  # the forest has about n edges
    if kind == "smooth_gs":
        return {"bytes": csr + block, "flops": T * sweep_g}
    off = m - n + 1
    flops = T * (sweep_g + sweep_p) + off * 6 * K
    if kind == "filter":
        return {"bytes": edges + 16 * m + 12 * n + 16 * n + 12 * n + 8 * off + 4 * int(case["budget"] * n), "flops": flops}
    if kind == "batch":
        return {"bytes": edges + 16 * m + 12 * n + 28 * n + m, "flops": flops}
    return {"bytes": edges + (csr if kind == "sparsify" else edges) + m, "flops": flops}


# ------------------------------------------------------------------------------------------------ 64-bit references

_M = (1 << 64) - 1


def _signed(x):
    x &= _M
    return x - (1 << 64) if x >> 63 else x


def _mix(x):
    """SplitMix64 of an int64 tensor holding 64-bit words."""
    def shr(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)
    z = x + _signed(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * _signed(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * _signed(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _block(n, K, seed):
    s0 = _mix(torch.tensor([_signed(seed)], dtype=torch.int64, device=DEV))
    o = _mix(s0 + torch.arange(n * K // 2, dtype=torch.int64, device=DEV) * _signed(0x9E3779B97F4A7C15))
    u1 = (((o >> 32) & 0xFFFFFFFF) + 1).double() * 2.0 ** -32
    u2 = ((o >> 8) & 0xFFFFFF).double() * 2.0 ** -24
    r, a = torch.sqrt(-2 * torch.log(u1)), 2 * math.pi * u2
    return torch.stack([r * torch.cos(a), r * torch.sin(a)], 1).reshape(n, K)


def _canonical(n, u, v, w):
    u, v = u.long(), v.long()
    keep = u != v
    u, v, w = u[keep], v[keep], w[keep].double()
    key, inv = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v), return_inverse=True)
    s = torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, inv, w)
    return key // n, key % n, s.float()


def _forest(n, u, v, w):
    """Maximum-weight spanning forest under (weight descending, edge id ascending), by Boruvka rounds."""
    m = u.numel()
    eid = torch.arange(m, device=DEV)
    key = (w.view(torch.int32).long() << 32) | (0xFFFFFFFF - eid)
    comp, mask = torch.arange(n, device=DEV), torch.zeros(m, dtype=torch.bool, device=DEV)
    while True:
        cu, cv = comp[u], comp[v]
        out = cu != cv
        if not bool(out.any()):
            return mask
        best = torch.zeros(n, dtype=torch.int64, device=DEV)
        for c in (cu, cv):
            best.scatter_reduce_(0, c[out], key[out], "amax")
        root = torch.nonzero(best > 0).reshape(-1)
        e = 0xFFFFFFFF - (best[root] & 0xFFFFFFFF)
        mask[e] = True
        parent = torch.arange(n, device=DEV)
        parent[root] = cu[e] + cv[e] - root
        me = torch.arange(n, device=DEV)
        parent = torch.where((parent[parent] == me) & (me < parent), me, parent)
        while True:
            up = parent[parent]
            if bool((up == parent).all()):
                break
            parent = up
        comp = parent[comp]


def _csr(n, u, v, w):
    """(row, column, weight) of both directions sorted by row and column, the matrix, and its row sums."""
    r, c, x = torch.cat([u, v]), torch.cat([v, u]), torch.cat([w, w]).double()
    order = torch.argsort(r * n + c)
    r, c, x = r[order], c[order], x[order]
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    deg = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, r, x)
    return r, c, x, torch.sparse_csr_tensor(ptr, c, x, size=(n, n)), deg


def _project(x):
    x = x - x.mean(0)
    rms = x.square().mean(0).sqrt()
    return x / torch.where(rms > 0, rms, torch.ones_like(rms))


def _smooth(n, u, v, w, x, steps, omega=0.7):
    _, _, _, A, deg = _csr(n, u, v, w)
    on = (deg > 0)[:, None]
    inv = torch.where(deg > 0, 1 / deg, deg)[:, None]
    for _ in range(steps):
        x = torch.where(on, (1 - omega) * x + omega * inv * (A @ x), x)
    return _project(x)


def _exact_filter(case, seed):
    n, u, v, w = _edges(case, seed)
    u, v, w = _canonical(n, u, v, w)
    tree = _forest(n, u, v, w)
    x = _block(n, case["K"], seed)
    xg = _smooth(n, u, v, w, x, case["steps"])
    xp = _smooth(n, u[tree], v[tree], w[tree], x, case["steps"])
    u, v, w = u[~tree], v[~tree], w[~tree].double()
    out = []
    for i in range(0, u.numel(), 1 << 19):
        p, q, ww = u[i:i + (1 << 19)], v[i:i + (1 << 19)], w[i:i + (1 << 19)]
        sg, sp = ww * (xg[p] - xg[q]).square().sum(1), ww * (xp[p] - xp[q]).square().sum(1)
        out.append((sp / (sg + 1e-30), sg, sp)[case["mode"]])
    return {"scores": torch.cat(out) if out else torch.empty(0, dtype=torch.float64, device=DEV), "selected": None}


def _colouring(n, r, c):
    """Jones-Plassmann: nodes that outrank their uncoloured neighbours take the smallest colour free around them."""
    rank = _mix(torch.arange(n, device=DEV) ^ 0x636F6C6F72) ^ (-1 << 63)  # unsigned order as signed
    colour = torch.full((n,), -1, dtype=torch.int64, device=DEV)
    low = torch.iinfo(torch.int64).min
    while bool((colour < 0).any()):
        free = colour < 0
        top = torch.full((n,), low, dtype=torch.int64, device=DEV)
        both = free[r] & free[c]
        top.scatter_reduce_(0, r[both], rank[c[both]], "amax")
        todo = free & (rank > top)
        before, k = colour.clone(), 0
        while bool(todo.any()):
            held = torch.zeros(n, dtype=torch.bool, device=DEV)
            held[r[before[c] == k]] = True
            now = todo & ~held
            colour[now] = k
            todo, k = todo & held, k + 1
    return colour


def _exact_gs(case, seed):
    n, u, v, w = _edges(case, seed)
    u, v, w = _canonical(n, u, v, w)
    r, c, x, _, deg = _csr(n, u, v, w)
    colour = _colouring(n, r, c)
    X = _block(n, case["K"], seed)
    X = X - X.mean(0)
    classes = []
    for k in range(int(colour.max()) + 1):
        e = colour[r] == k
        rows = torch.nonzero((colour == k) & (deg > 0)).reshape(-1)
        at = torch.zeros(n, dtype=torch.int64, device=DEV)
        at[rows] = torch.arange(rows.numel(), device=DEV)
        cnt = torch.bincount(at[r[e]], minlength=rows.numel())
        ptr = torch.zeros(rows.numel() + 1, dtype=torch.int64, device=DEV)
        ptr[1:] = torch.cumsum(cnt, 0)
        classes.append((rows, torch.sparse_csr_tensor(ptr, c[e], x[e], size=(rows.numel(), n)), 1 / deg[rows][:, None]))
    for _ in range(case["steps"]):
        for rows, A, inv in classes:
            X[rows] = inv * (A @ X)
    return {"x": _project(X)}


def _exact_laplacian(case, seed):
    n, u, v, w = _edges(case, seed)
    _, _, x, _, deg = _csr(n, *_canonical(n, u, v, w))
    return {"row_ptr": None, "col": None, "val": x, "eid": None, "deg": deg}


def _network(theta, x):
    a, b = NFEAT * HID, NFEAT * HID + HID
    h = torch.relu(x @ theta[:a].reshape(NFEAT, HID) + theta[a:b])
    h = torch.relu(h @ theta[b:b + HID * HID].reshape(HID, HID) + theta[b + HID * HID:b + HID * HID + HID])
    return h @ theta[-HID - 1:-1] + theta[-1]


def _exact_mlp(case, seed):
    theta, x, t = (a.double() for a in _mlp_inputs(case, seed))
    if case["kind"] == "mlp_forward":
        return {"y": torch.cat([_network(theta, x[i:i + (1 << 20)]) for i in range(0, x.shape[0], 1 << 20)])}
    theta.requires_grad_(True)
    total, rows = 0.0, x.shape[0]
    for i in range(0, rows, 1 << 19):
        part = (_network(theta, x[i:i + (1 << 19)]) - t[i:i + (1 << 19)]).square().sum() / rows
        part.backward()
        total += float(part.detach())
    return {"grad": theta.grad, "loss": total}


def exact(case, seed):
    kind = case["kind"]
    if kind == "filter":
        return _exact_filter(case, seed)
    if kind == "smooth_gs":
        return _exact_gs(case, seed)
    if kind == "laplacian":
        return _exact_laplacian(case, seed)
    if kind in ("mlp_forward", "mlp_gradient"):
        return _exact_mlp(case, seed)
    if kind == "end_to_end":
        return {"u": None, "v": None, "w": _canonical(*_edges(case, seed))[2].double(), "mask": None, "count": None}
    return None  # masks and maps: whole numbers
