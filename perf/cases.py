"""What a user of this framework has it do, as timed cases.

A case is a dict of plain values.  Whole reductions (a graph created from its
edge list, then the level loop, then the reduced graph and the composed map
read) stand beside the single steps a program calls by themselves: smoothing,
Gauss-Seidel smoothing, affinity, the spectral-mismatch loss and its gradient,
edge scaling, the multilevel eigensolver and the reduced data set.

Graphs are made on the GPU from the seed alone, in the shapes of the
repository's named workloads: 2-D grids and 3-D 7-point meshes with log-normal
weights, k-nearest-neighbour graphs of Gaussian-mixture points, and power-law
(Chung-Lu) graphs with unit weights.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1812_08942_gb300 as gr

DEV = "cuda"
PREC = {"f64": (torch.float64, gr.GR_F64, 8), "f32": (torch.float32, gr.GR_F32, 4),
        "bf16": (torch.bfloat16, gr.GR_BF16, 2)}


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest whole reduction: a 64 x 64 grid in FP64 (launches and host waits count)
        dict(name="reduce_grid_f64", kind="reduce", graph="mesh", a=64, b=64, c=1, K=8, sweeps=5, prec="f64",
             target=1024),
        # the headline reduction: a 128^3 mesh, 24 test vectors, down to n / 64
        dict(name="reduce_mesh_f32", kind="reduce", graph="mesh", a=128, b=128, c=128, K=24, sweeps=8, prec="f32",
             target=32768),
        # a data set's neighbour graph: 200,000 points in 10-D, 10 neighbours each
        dict(name="reduce_knn_f32", kind="reduce", graph="knn", n=200000, dim=10, k=10, K=16, sweeps=5, prec="f32",
             target=6250),
        # a collaboration network's shape: 434,000 nodes, 16 M edges, hubs of degree 1,200
        dict(name="reduce_powerlaw_f32", kind="reduce", graph="powerlaw", n=434000, m=16000000, K=16, sweeps=5,
             prec="f32", target=13000),
        # smoothing by itself where accuracy comes first: FP64 on a 64^3 mesh
        dict(name="smooth_mesh_f64", kind="smooth", graph="mesh", a=64, b=64, c=64, K=24, sweeps=8, prec="f64"),
        # smoothing by itself where memory comes first: BF16 storage on a neighbour graph
        dict(name="smooth_knn_bf16", kind="smooth", graph="knn", n=200000, dim=10, k=10, K=16, sweeps=5,
             prec="bf16"),
        # the other relaxation: colouring and multicolour Gauss-Seidel on a ragged mesh
        dict(name="gauss_seidel_mesh_f32", kind="gauss_seidel", graph="mesh", a=101, b=89, c=75, K=16, sweeps=5,
             prec="f32"),
        # affinities and distances of given vectors
        dict(name="affinity_mesh_f32", kind="affinity", graph="mesh", a=127, b=119, c=103, K=24, prec="f32"),
        # loss and gradient with respect to the reduced graph's weights, through autograd
        dict(name="loss_mesh", kind="loss", graph="mesh", a=128, b=128, c=128, cell=4.0, K=24, sweeps=5),
        # ten iterations of edge scaling on a reduced mesh
        dict(name="scale_edges_mesh", kind="scale", graph="mesh", a=96, b=80, c=64, cell=4.0, K=16, sweeps=5,
             iters=10),
        # eight eigenvectors of a mesh through a hierarchy down to about 1,000 nodes
        dict(name="eigensolve_mesh", kind="eigensolve", graph="mesh", a=128, b=128, c=128, coarsest=1000, k=8,
             iters=10, mass=1, normalized=0),
        # a data set's features carried to the reduced nodes
        dict(name="dataset_mesh", kind="dataset", graph="mesh", a=128, b=128, c=128, d=16, prec="f32", mean=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh_sides(rng, lo, hi):
    """Three sides of about lo .. hi nodes in all, none a multiple of the other by design."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    s = n ** (1.0 / 3.0)
    a = max(2, int(round(s * rng.uniform(0.7, 1.4))))
    b = max(2, int(round(s * rng.uniform(0.7, 1.4))))
    return dict(graph="mesh", a=a, b=b, c=max(2, int(n / (a * b))))


def _any_graph(rng, side=24):
    g = rng.choice(["grid", "mesh", "knn", "powerlaw"])
    if g == "grid":
        return dict(graph="mesh", a=_log_int(rng, side, 700), b=_log_int(rng, side, 700), c=1)
    if g == "mesh":
        return _mesh_sides(rng, 20000, 2000000)
    if g == "knn":
        return dict(graph="knn", n=_log_int(rng, 10000, 200000), dim=rng.choice([8, 10, 16]),
                    k=rng.choice([7, 10, 15]))
    n = _log_int(rng, 8000, 434000)
    return dict(graph="powerlaw", n=n, m=int(n * rng.uniform(20.0, 36.0)))


def draw(rng):
    kind = rng.choice(["reduce", "reduce", "reduce", "smooth", "gauss_seidel", "affinity", "loss", "scale",
                       "eigensolve", "dataset"])
    K = rng.choice([4, 8, 16, 24, 32])
    if kind == "reduce":
        c = dict(kind=kind, K=rng.choice([8, 16, 24]), sweeps=rng.choice([4, 5, 6, 8]),
                 prec=rng.choice(["f32", "f32", "f64"]), **_any_graph(rng))
        c["target"] = max(16, _nodes(c) // rng.choice([4, 16, 32, 64]))
        return c
    if kind == "smooth":
        return dict(kind=kind, K=K, sweeps=rng.choice([3, 5, 8]), prec=rng.choice(["f64", "f32", "bf16"]),
                    **_any_graph(rng))
    if kind == "gauss_seidel":
        return dict(kind=kind, K=K, sweeps=rng.choice([2, 5]), prec=rng.choice(["f64", "f32"]),
                    **_mesh_sides(rng, 8000, 1000000))
    if kind == "affinity":
        return dict(kind=kind, K=K, prec=rng.choice(["f64", "f32", "bf16"]), **_any_graph(rng, 150))
    if kind == "loss":
        return dict(kind=kind, K=K, sweeps=rng.choice([2, 5]), cell=rng.uniform(2.2, 6.0),
                    **_mesh_sides(rng, 8000, 2000000))
    if kind == "scale":
        return dict(kind=kind, K=K, sweeps=rng.choice([2, 5]), cell=rng.uniform(2.5, 6.0), iters=rng.choice([4, 10]),
                    **_mesh_sides(rng, 8000, 500000))
    if kind == "eigensolve":
        # (ratio cut with each level's own mass divides by nearly vanishing
        # diagonals on weighted meshes: its results are not reproducible digits)
        mass, normalized = rng.choice([(1, 0), (1, 1), (0, 1)])
        return dict(kind=kind, coarsest=rng.choice([300, 700, 1000]), k=rng.choice([3, 4, 8]),
                    iters=rng.choice([5, 10]), mass=mass, normalized=normalized, **_mesh_sides(rng, 30000, 2000000))
    return dict(kind=kind, d=rng.choice([1, 3, 10, 16, 24]), prec=rng.choice(["f64", "f32"]), mean=rng.choice([0, 1]),
                **_mesh_sides(rng, 8000, 2000000))


# ---------------------------------------------------------------------------
# Graphs (canonical edge lists on the GPU)
# ---------------------------------------------------------------------------
def _nodes(case):
    return case["a"] * case["b"] * case["c"] if case["graph"] == "mesh" else case["n"]


def _edges(case):
    if case["graph"] == "mesh":
        a, b, c = case["a"], case["b"], case["c"]
        return (a - 1) * b * c + a * (b - 1) * c + a * b * (c - 1)
    return case["m"] if case["graph"] == "powerlaw" else int(0.58 * case["n"] * case["k"])


def _generator(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _mesh(case, seed):
    a, b, c = case["a"], case["b"], case["c"]
    n = a * b * c
    p = torch.arange(n, device=DEV)
    i, j, k = p % a, (p // a) % b, p // (a * b)
    v = torch.stack([p + 1, p + a, p + a * b], 1)
    keep = torch.stack([i < a - 1, j < b - 1, k < c - 1], 1)
    u = p[:, None].expand(-1, 3)[keep].to(torch.int32)
    v = v[keep].to(torch.int32)
    w = torch.randn(u.numel(), dtype=torch.float64, device=DEV, generator=_generator(seed, 1)).exp_()
    return n, u, v, w


def _unique_pairs(n, lo, hi, w=None):
    key = lo * n + hi
    if w is None:
        return torch.unique(key), None
    key, order = torch.sort(key, stable=True)
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    return key[first], w[order][first]


def _knn(case, seed):
    """Exact neighbours within each of ten Gaussian components (which lie far
    apart), symmetrised, weights exp(-d^2 / median(d)^2); a random
    surplus is dropped so that exactly _edges(case) remain."""
    n, dim, k, ncomp = case["n"], case["dim"], case["k"], 10
    g = _generator(seed, 2)
    pts = torch.randn(n, dim, device=DEV, generator=g)
    comp = torch.randint(0, ncomp, (n,), device=DEV, generator=g)
    src, dst, dist = [], [], []
    for q in range(ncomp):
        ids = torch.nonzero(comp == q).flatten()
        x = pts[ids]
        sq = (x * x).sum(1)
        kk = min(k, ids.numel() - 1)
        for s in range(0, ids.numel(), 8192):
            e = min(s + 8192, ids.numel())
            d2 = sq[s:e, None] - 2.0 * (x[s:e] @ x.T) + sq[None, :]
            d2[torch.arange(e - s, device=DEV), torch.arange(s, e, device=DEV)] = math.inf
            val, nb = torch.topk(d2, kk, dim=1, largest=False)
            src.append(ids[s:e, None].expand(-1, kk).flatten())
            dst.append(ids[nb].flatten())
            dist.append(val.clamp_min_(0).sqrt_().flatten().double())
    src, dst, dist = torch.cat(src), torch.cat(dst), torch.cat(dist)
    w = torch.exp(-(dist / dist.median()) ** 2).clamp_min_(1e-300)
    key, w = _unique_pairs(n, torch.minimum(src, dst), torch.maximum(src, dst), w)
    keep = torch.argsort(torch.rand(key.numel(), dtype=torch.float64, device=DEV, generator=g))
    keep = torch.sort(keep[:_edges(case)]).values
    key, w = key[keep], w[keep]
    return n, (key // n).to(torch.int32), (key % n).to(torch.int32), w


def _powerlaw(case, seed):
    """Chung-Lu: expected degrees c (1 + i / i0)^(-2/3), c = 1,200 at most a
    quarter of n, i0 solved for the mean degree; exactly m unit edges."""
    n, m = case["n"], case["m"]
    g = _generator(seed, 3)
    top, mean = min(1200.0, n / 4.0), 2.0 * m / n
    i = torch.arange(n, dtype=torch.float64, device=DEV)
    lo, hi = math.log(1e-3), math.log(1e3 * n)
    for _ in range(50):
        mid = 0.5 * (lo + hi)
        if float((top * (1.0 + i / math.exp(mid)) ** (-2.0 / 3.0)).mean()) < mean:
            lo = mid
        else:
            hi = mid
    cdf = torch.cumsum((1.0 + i / math.exp(0.5 * (lo + hi))) ** (-2.0 / 3.0), 0)
    cdf /= cdf[-1].clone()
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    need = m
    while need > 0:
        cnt = int(need * 1.15) + 1024
        r = torch.rand(2, cnt, dtype=torch.float64, device=DEV, generator=g)
        a, b = torch.searchsorted(cdf, r, right=True).clamp_max_(n - 1)
        ok = a != b
        key, _ = _unique_pairs(n, torch.minimum(a, b)[ok], torch.maximum(a, b)[ok])
        keys = torch.unique(torch.cat([keys, key]))
        need = m - keys.numel()
    if need < 0:  # drop a random surplus
        order = torch.argsort(torch.rand(keys.numel(), dtype=torch.float64, device=DEV, generator=g))
        keys = torch.sort(keys[order[:m]]).values
    return n, (keys // n).to(torch.int32), (keys % n).to(torch.int32), torch.ones(m, dtype=torch.float64, device=DEV)


def _graph(case, seed):
    return {"mesh": _mesh, "knn": _knn, "powerlaw": _powerlaw}[case["graph"]](case, seed)


# ---------------------------------------------------------------------------
# Aggregates of a mesh: Voronoi cells of jittered block centres (irregular
# cells with about 14 neighbours each, as aggregation makes them), the same for
# every seed, so that a case's reduced graph keeps its size
# ---------------------------------------------------------------------------
def _voronoi(pos, dims, cell, gen):
    nb = [max(1, int(math.ceil(d / cell))) for d in dims]
    step = torch.tensor([d / q for d, q in zip(dims, nb)], device=DEV)
    size = torch.tensor(nb, device=DEV)
    blk = torch.stack(torch.meshgrid(*[torch.arange(q, device=DEV) for q in nb], indexing="ij"), -1).reshape(-1, 3)
    seeds = (blk + 0.1 + 0.8 * torch.rand(blk.shape, device=DEV, generator=gen)) * step
    home = torch.minimum((pos / step).long(), size - 1)
    best = torch.full((pos.shape[0],), math.inf, device=DEV)
    own = torch.zeros(pos.shape[0], dtype=torch.int64, device=DEV)
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                q = home + torch.tensor([dx, dy, dz], device=DEV)
                ok = ((q >= 0) & (q < size)).all(1)
                q = torch.minimum(q.clamp_min(0), size - 1)
                s = (q[:, 0] * nb[1] + q[:, 1]) * nb[2] + q[:, 2]
                d = ((seeds[s] - pos) ** 2).sum(1)
                better = ok & (d < best)
                best = torch.where(better, d, best)
                own = torch.where(better, s, own)
    used, agg = torch.unique(own, return_inverse=True)
    return agg.to(torch.int32), used.numel(), seeds[used]


def _mesh_maps(case, cells):
    a, b, c = case["a"], case["b"], case["c"]
    p = torch.arange(a * b * c, device=DEV)
    pos = torch.stack([p % a, (p // a) % b, p // (a * b)], 1).float() + 0.5
    gen = _generator(0, 4)
    maps = []
    for cell in cells:
        agg, nc, pos = _voronoi(pos, (a, b, c), cell, gen)
        maps.append((agg, nc))
    return maps


def _cells_to(case, target):
    last = max(2.0, (_nodes(case) / target) ** (1.0 / 3.0))
    cells = [2.0]
    while cells[-1] * 1.5 < last:
        cells.append(min(cells[-1] * 2.0, last))
    return cells


def _coarse_edges(agg, nc, u, v, w):
    """P^T L P as a canonical edge list, in plain torch."""
    a, b = agg[u.long()].long(), agg[v.long()].long()
    ok = a != b
    key, inv = torch.unique(torch.minimum(a, b)[ok] * nc + torch.maximum(a, b)[ok], return_inverse=True)
    wc = torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, inv, w[ok])
    return (key // nc).to(torch.int32), (key % nc).to(torch.int32), wc


def _vectors(n, u, v, w, K, seed, sweeps=3):
    """K random vectors relaxed a little on the graph, centred, unit norm (FP64
    numbers rounded to 24 bits, so that the order of the sums does not show)."""
    x = torch.randn(n, K, dtype=torch.float64, device=DEV, generator=_generator(seed, 5))
    A = _Adjacency(n, u, v, w)
    for _ in range(sweeps):
        x = A.jacobi(x, 0.7)
        x -= x.mean(0)
        x /= x.norm(dim=0)
    return x.float().double()


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    n, u, v, w = _graph(case, seed)
    s = dict(case=case, n=n, seed=int(seed) & 0x7FFFFFFF)
    if kind == "reduce":
        s.update(u=u, v=v, w=w, params=gr.ReduceParams(
            K=case["K"], sweeps=case["sweeps"], seed=s["seed"], prec=PREC[case["prec"]][1],
            final_target=case["target"]))
        # the result's buffers, kept across passes as a program that reduces many graphs keeps them
        s["out"] = tuple(torch.zeros_like(t) for t in (u, v, w))
        return s
    s["g"] = gr.graph_reduce_create(n, u, v, w)
    if kind in ("smooth", "gauss_seidel"):
        s["X"] = torch.empty(n, case["K"], dtype=PREC[case["prec"]][0], device=DEV)
    elif kind == "affinity":
        dt = PREC[case["prec"]][0]
        s["X"] = _vectors(n, u, v, w, case["K"], seed).to(dt)
        out = torch.float64 if dt == torch.float64 else torch.float32
        s["d"] = torch.empty(u.numel(), dtype=out, device=DEV)
        s["a"] = torch.empty_like(s["d"])
    elif kind in ("loss", "scale"):
        (agg, nc), = _mesh_maps(case, [case["cell"]])
        s["agg"] = agg
        s["coarse"] = gr.graph_reduce_coarsen(s["g"], agg, nc)
        s["X"] = _vectors(n, u, v, w, case["K"], seed).float()
        s["w"] = gr.graph_reduce_get_edges(s["coarse"])[2].float()
        if kind == "scale":
            s["eta"] = _step_size(n, u, v, w, agg, nc, s["X"], case["sweeps"])
    else:
        cells = _cells_to(case, case["coarsest"]) if kind == "eigensolve" else [2.0, 4.0]
        s["levels"] = [s["g"]]
        for agg, nc in _mesh_maps(case, cells):
            s["levels"].append(gr.graph_reduce_coarsen(s["levels"][-1], agg, nc))
        if kind == "dataset":
            s["F"] = torch.randn(n, case["d"], dtype=PREC[case["prec"]][0], device=DEV,
                                 generator=_generator(seed, 6))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "reduce":
        g = gr.graph_reduce_create(s["n"], s["u"], s["v"], s["w"])
        levels, _ = gr.graph_reduce_multilevel(g, s["params"], want_stats=False)
        gr.graph_reduce_get_edges(levels[-1], out=s["out"])
        u, v, w = s["out"]
        return {"labels": gr.graph_reduce_compose_maps(levels), "u": u, "v": v, "w": w,
                "nodes": levels[-1].n, "edges": levels[-1].m}
    if kind == "smooth":
        return gr.graph_reduce_smooth(s["g"], s["X"], case["sweeps"], seed=s["seed"])
    if kind == "gauss_seidel":
        colour, _ = gr.graph_reduce_colour(s["g"], s["seed"])
        X = gr.graph_reduce_smooth_gs(s["g"], s["X"], case["sweeps"], seed=s["seed"], colour_seed=s["seed"])
        return {"colour": colour, "X": X}
    if kind == "affinity":
        gr.graph_reduce_affinity(s["g"], s["X"], s["d"], s["a"])
        return {"d": s["d"], "a": s["a"]}
    if kind == "loss":
        w = s["w"].detach().requires_grad_(True)
        loss = gr.spectral_mismatch_loss(w, s["g"], s["coarse"], s["agg"], s["X"], case["sweeps"])
        return {"loss": loss.detach(), "grad": torch.autograd.grad(loss, w)[0]}
    if kind == "scale":
        w, hist = gr.graph_reduce_scale_edges(s["g"], s["coarse"], s["agg"], s["X"], s["w"].clone(), case["sweeps"],
                                              eta_max=s["eta"], eps=0.0, kmax=case["iters"])
        return {"w": w, "history": _history(hist, case["iters"])}
    if kind == "eigensolve":
        U, lam, rq = gr.graph_reduce_eigensolve(s["levels"], case["k"], normalized=bool(case["normalized"]),
                                                iters=case["iters"], galerkin_mass=bool(case["mass"]))
        return {"U": U, "lambda": lam, "rayleigh": rq}
    return gr.graph_reduce_reduce_data(s["levels"][1:], s["F"], mean=bool(case["mean"]))


def _history(hist, iters):
    """(loss, lambda_1) per iteration as the single-precision record a program plots."""
    out = np.zeros((iters, 2), np.float32)
    out[:len(hist)] = hist
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without: inputs read once, outputs written once
# ---------------------------------------------------------------------------
def work(case):
    kind, n, m = case["kind"], _nodes(case), _edges(case)
    graph = 16.0 * m  # u, v int32 and w float64
    if kind == "reduce":
        K, S = case["K"], case["sweeps"]
        nc = case["target"]
        mc = min(m, 8 * nc)
        return {"bytes": graph + 4.0 * n + 16.0 * mc, "flops": S * (4.0 * m * K + 6.0 * n * K) + 12.0 * m * K}
    if kind in ("smooth", "gauss_seidel"):
        K, S, sz = case["K"], case["sweeps"], PREC[case["prec"]][2]
        return {"bytes": graph + float(n) * K * sz + (4.0 * n if kind == "gauss_seidel" else 0.0),
                "flops": S * (4.0 * m * K + 6.0 * n * K)}
    if kind == "affinity":
        K, sz = case["K"], PREC[case["prec"]][2]
        return {"bytes": 8.0 * m + float(n) * K * sz + 2.0 * m * max(sz, 4), "flops": 12.0 * m * K}
    if kind in ("loss", "scale"):
        K, S = case["K"], case["sweeps"]
        nc = n / case["cell"] ** 3
        mc = min(m, 7 * nc)
        it = case["iters"] if kind == "scale" else 1
        return {"bytes": graph + 4.0 * n + 4.0 * n * K + 12.0 * mc + 8.0 * mc,
                "flops": 4.0 * m * K + 4.0 * n * K + it * (3 * S + 3) * 4.0 * mc * K}
    if kind == "eigensolve":
        k = case["k"]
        return {"bytes": 8.0 / 7.0 * (graph + 4.0 * n) + 8.0 * n * k,
                "flops": 8.0 / 7.0 * case["iters"] * (4.0 * m * k + 3.0 * n * k) + 2.0 * n * k * k + 5.0 * m * k}
    sz = PREC[case["prec"]][2]
    return {"bytes": float(n) * case["d"] * sz * (1.0 + 1.0 / 64.0) + 4.0 * n * 9.0 / 8.0, "flops": float(n) * case["d"]}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------
class _Adjacency:
    """Symmetric adjacency as slots (row, col, w) and the degrees, FP64."""

    def __init__(self, n, u, v, w):
        self.n = n
        self.r = torch.cat([u, v]).long()
        self.c = torch.cat([v, u]).long()
        self.w = torch.cat([w, w])
        self.deg = torch.zeros(n, dtype=torch.float64, device=DEV).index_add(0, self.r, self.w)

    def apply(self, x):
        out = torch.zeros_like(x)
        step = max(1, (1 << 27) // max(1, x.shape[1]))
        for s in range(0, self.r.numel(), step):
            t = slice(s, s + step)
            out = out.index_add(0, self.r[t], self.w[t, None] * x[self.c[t]])
        return out

    def jacobi(self, x, omega):
        has = (self.deg > 0)[:, None]
        z = torch.where(has, self.apply(x) / torch.where(has, self.deg[:, None], torch.ones_like(x[:, :1])), x)
        return (1.0 - omega) * x + omega * z


def _mix(z):
    """The finaliser of SplitMix64 (Steele, Lea, Flood 2014) on int64 bit patterns."""
    def shr(x, k):
        return (x >> k) & ((1 << (64 - k)) - 1)

    z = (z ^ shr(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ shr(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ shr(z, 31)


def _splitmix(seed, c):
    return _mix(seed + (c + 1) * (0x9E3779B97F4A7C15 - (1 << 64)))


def _test_vectors(n, K, seed):
    z = _splitmix(seed, torch.arange(n * K, device=DEV))
    t = ((z >> 11) & ((1 << 53) - 1)) - (1 << 52)
    return (t.double() * 2.0 ** -52).reshape(n, K)


def _unit(x):
    x = x - x.mean(0)
    return x / x.norm(dim=0)


def _colouring(A, seed):
    """Greedy colouring in descending priority, by rounds of local maxima."""
    prio = _splitmix(seed, torch.arange(A.n, device=DEV) + (1 << 62)) ^ (-(1 << 63))  # unsigned order as signed
    colour = torch.full((A.n,), -1, dtype=torch.int64, device=DEV)
    beats = (prio[A.c] > prio[A.r]) | ((prio[A.c] == prio[A.r]) & (A.c > A.r))
    while bool((colour < 0).any()):
        open_ = colour < 0
        blocked = torch.zeros(A.n, dtype=torch.bool, device=DEV)
        t = beats & open_[A.c]
        blocked[A.r[t]] = True
        now = open_ & ~blocked
        t = now[A.r] & ~open_[A.c]
        used = torch.zeros(A.n, 64, dtype=torch.bool, device=DEV)
        used[A.r[t], colour[A.c[t]]] = True
        first = torch.where(used, 64, torch.arange(64, device=DEV)).amin(1)
        colour = torch.where(now, first, colour)
    return colour


def _quotients(A, u, v, w, x, mass):
    d = x[u] - x[v]
    mu = (mass[:, None] * x).sum(0) / mass.sum()
    return (w[:, None] * d * d).sum(0) / (mass[:, None] * (x - mu) ** 2).sum(0)


class _Loss:
    """The spectral-mismatch loss in FP64, differentiable in the reduced weights."""

    def __init__(self, n, u, v, w, agg, nc, X, sweeps):
        self.uc, self.vc, self.wc = _coarse_edges(agg, nc, u, v, w)
        self.ul, self.vl = self.uc.long(), self.vc.long()
        X = X.double()
        step = 1 << 20
        num = sum((w[s:s + step, None] * (X[u[s:s + step].long()] - X[v[s:s + step].long()]) ** 2).sum(0)
                  for s in range(0, u.numel(), step))
        self.Rf = num / (X * X).sum(0)
        self.mass = torch.zeros(nc, dtype=torch.float64, device=DEV).index_add(0, agg.long(),
                                                                               torch.ones_like(X[:, 0]))
        self.y0 = torch.zeros(nc, X.shape[1], dtype=torch.float64, device=DEV).index_add(0, agg.long(), X)
        self.y0 = self.y0 / self.mass[:, None]
        self.nc, self.sweeps = nc, sweeps

    def __call__(self, wc):
        A = _Adjacency(self.nc, self.uc, self.vc, wc)
        y = self.y0
        for _ in range(self.sweeps):
            y = A.jacobi(y, 0.7)
        Rc = _quotients(A, self.ul, self.vl, wc, y, self.mass)
        return ((Rc / self.Rf - 1.0) ** 2).mean()

    def gradient(self, wc):
        wc = wc.detach().requires_grad_(True)
        loss = self(wc)
        return loss.detach(), torch.autograd.grad(loss, wc)[0]


def _step_size(n, u, v, w, agg, nc, X, sweeps):
    """A step whose first update moves an edge by at most 5 % of the mean weight (3 digits)."""
    L = _Loss(n, u, v, w, agg, nc, X, sweeps)
    wc = L.wc.float().double()
    return float("%.2e" % (0.05 * float(wc.mean()) / float(L.gradient(wc)[1].abs().max())))


def _scale_exact(L, w, eta_max, iters, alpha=0.5, delta_bar=0.5):
    def degrees(x):
        return torch.zeros(L.nc, dtype=torch.float64, device=DEV).index_add(0, torch.cat([L.ul, L.vl]),
                                                                            torch.cat([x, x]))

    dG = degrees(w)
    dP, dw, lam1, eta = dG, torch.zeros_like(w), 1.0, eta_max
    losses, lams = [], []
    for k in range(iters):
        loss, grad = L.gradient(w)
        loss = float(loss)
        if k > 0 and losses[-1] < loss:
            break
        bound = lam1 * delta_bar ** (1.0 / iters)
        d = (alpha * dw - eta * grad).clamp_min(0.0)
        p, q = L.ul, L.vl
        low = torch.minimum(dG[p] / (dP[p] + d), dG[q] / (dP[q] + d)) <= bound
        cap = torch.minimum(dG[p] / bound - dP[p], dG[q] / bound - dP[q]).clamp_min(0.0)
        dw = torch.where(low, cap, d)
        w = w + dw
        dP = degrees(w)
        has = dP > 0
        lam1 = float((dG[has] / dP[has]).min())
        losses.append(loss)
        lams.append(lam1)
        eta = loss / losses[0] * eta_max
    return w, losses, lams


def _eigen_exact(case, seed, n, u, v, w):
    graphs, maps = [(n, u, v, w)], _mesh_maps(case, _cells_to(case, case["coarsest"]))
    for agg, nc in maps:
        _, a, b, x = graphs[-1]
        graphs.append((nc,) + _coarse_edges(agg, nc, a, b, x))
    A = [_Adjacency(*g) for g in graphs]
    own = [g.deg if case["normalized"] else torch.ones_like(g.deg) for g in A]
    mass = own[:1]
    for l, (agg, nc) in enumerate(maps):
        mass.append(torch.zeros_like(own[l + 1]).index_add(0, agg.long(), mass[-1]) if case["mass"] else own[l + 1])
    nc = graphs[-1][0]
    Lc = torch.diag(A[-1].deg).index_put((A[-1].r, A[-1].c), -A[-1].w, accumulate=True)
    sq = mass[-1].rsqrt()
    lam, Y = torch.linalg.eigh((sq[:, None] * Lc * sq[None, :]).cpu())
    lam = lam[:case["k"]].to(DEV)
    Y = sq[:, None] * Y[:, :case["k"]].to(DEV)
    for l in range(len(maps) - 1, -1, -1):
        Y = Y[maps[l][0].long()]
        diag = A[l].deg[:, None] - lam * mass[l][:, None]
        for _ in range(case["iters"]):
            Y = torch.where(diag > 0, 0.3 * Y + 0.7 * A[l].apply(Y) / diag, Y)
    for i in range(case["k"]):
        for j in range(i):
            Y[:, i] -= (Y[:, i] @ Y[:, j]) * Y[:, j]
        Y[:, i] /= Y[:, i].norm()
    d = Y[u.long()] - Y[v.long()]
    return lam.cpu().numpy(), ((w[:, None] * d * d).sum(0) / (own[0][:, None] * Y * Y).sum(0)).cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "reduce":  # a matching decides every output: whole numbers, and sums over them
        return None
    n, u, v, w = _graph(case, seed)
    s = int(seed) & 0x7FFFFFFF
    if kind in ("smooth", "gauss_seidel"):
        A = _Adjacency(n, u, v, w)
        x = _unit(_test_vectors(n, case["K"], s))
        if kind == "smooth":
            for _ in range(case["sweeps"]):
                x = _unit(A.jacobi(x, 0.7))
            return x
        colour = _colouring(A, s)
        parts = []
        for c in range(int(colour.max()) + 1):
            t = colour[A.r] == c
            rows = torch.nonzero((colour == c) & (A.deg > 0)).flatten()
            parts.append((A.r[t], A.c[t], A.w[t], rows))
        for _ in range(case["sweeps"]):
            for r, c, ww, rows in parts:
                z = torch.zeros_like(x).index_add(0, r, ww[:, None] * x[c])
                x[rows] = 0.3 * x[rows] + 0.7 * z[rows] / A.deg[rows, None]
            x = _unit(x)
        return {"colour": colour.to(torch.int32), "X": x}
    if kind == "affinity":
        X = _vectors(n, u, v, w, case["K"], seed).to(PREC[case["prec"]][0]).double()
        p, q = X[u.long()], X[v.long()]
        hp, hq = p / p.norm(dim=1, keepdim=True), q / q.norm(dim=1, keepdim=True)
        d = 0.25 * ((hp - hq) ** 2).sum(1) * ((hp + hq) ** 2).sum(1)
        return {"d": d, "a": (p * q).sum(1) ** 2 / ((p * p).sum(1) * (q * q).sum(1))}
    if kind in ("loss", "scale"):
        (agg, nc), = _mesh_maps(case, [case["cell"]])
        X = _vectors(n, u, v, w, case["K"], seed).float()
        L = _Loss(n, u, v, w, agg, nc, X, case["sweeps"])
        wc = L.wc.float().double()
        if kind == "loss":
            loss, grad = L.gradient(wc)
            return {"loss": loss, "grad": grad}
        eta = _step_size(n, u, v, w, agg, nc, X, case["sweeps"])
        wc, losses, lams = _scale_exact(L, wc, eta, case["iters"])
        return {"w": wc, "history": _history(list(zip(losses, lams)), case["iters"]).astype(np.float64)}
    if kind == "eigensolve":
        lam, rq = _eigen_exact(case, seed, n, u, v, w)
        return {"U": None, "lambda": lam, "rayleigh": rq}  # eigenvectors: up to the sign of a column
    label = torch.arange(n, device=DEV)
    for agg, nc in _mesh_maps(case, [2.0, 4.0]):
        label = agg.long()[label]
    F = torch.randn(n, case["d"], dtype=PREC[case["prec"]][0], device=DEV, generator=_generator(seed, 6)).double()
    out = torch.zeros(nc, case["d"], dtype=torch.float64, device=DEV).index_add(0, label, F)
    if case["mean"]:
        out = out / torch.bincount(label, minlength=nc)[:, None]
    return out
