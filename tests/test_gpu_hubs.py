"""Graphs with hubs, whose rows one lane or one thread would walk: the sums stay
those of short chains, the results those of the oracle or of plain FP64."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _hubs(n, mean, hubs, hub_deg, seed, at="first"):
    """Random edges and hubs: at the first nodes (upper edges) or the last ones (lower edges)."""
    rng = np.random.default_rng(seed)
    m = n * mean // 2
    a, b = rng.integers(0, n, m), rng.integers(0, n, m)
    for h in range(hubs):
        a = np.concatenate([a, np.full(hub_deg, h if at == "first" else n - 1 - h)])
        b = np.concatenate([b, rng.choice(n, hub_deg, replace=False)])
    keep = a != b
    u, v, w = W.canonicalize(n, a[keep], b[keep], rng.uniform(0.1, 2.0, int(keep.sum())))
    return W.Graph(n, u, v, w)


@pytest.mark.parametrize("K", [4, 24, 32])
@pytest.mark.parametrize("at,hub_deg,mean", [("first", 250000, 4), ("last", 250000, 4), ("first", 65, 4),
                                             ("first", 64, 1), ("first", 3000, 80)])
def test_fine_quotients(gpu_lib, K, at, hub_deg, mean):
    """R_f of FP32 vectors within 1e-6 of FP64: chains of some 64 FP32
    additions, then of a few hundred block sums (random signs of their
    roundings: sqrt(64 + 300) 2^-24 = 1.2e-6 for one lane, and 29,000 lanes)."""
    gr = gpu_lib
    n = 260000 if hub_deg > 3000 else 20000
    g = _hubs(n, mean, 2, hub_deg, 3, at)
    F = gr.graph_reduce_create(n, g.u, g.v, g.w)
    agg = torch.from_numpy((np.arange(n) // 16).astype(np.int32)).to(DEV)
    nc = -(-n // 16)
    C = gr.graph_reduce_coarsen(F, agg, nc)
    X = torch.randn(n, K, device=DEV, generator=torch.Generator(device=DEV).manual_seed(K))
    w = gr.graph_reduce_get_edges(C)[2].float()
    saved = gr.graph_reduce_loss_fwd(F, C, agg, X, w, 0)[1]
    X = X.double()
    u, v, ew = (torch.from_numpy(x).to(DEV) for x in (g.u, g.v, g.w))
    num = torch.zeros(K, dtype=torch.float64, device=DEV)
    for s in range(0, u.numel(), 1 << 18):
        t = slice(s, s + (1 << 18))
        num += (ew[t, None] * (X[u[t].long()] - X[v[t].long()]) ** 2).sum(0)
    ref = num / (X * X).sum(0)
    got = saved[nc * K:nc * K + K].double()
    assert ((got - ref).abs() / ref).max().item() <= 1e-6


@pytest.mark.parametrize("K,S", [(4, 2), (8, 0), (24, 1), (32, 2)])
@pytest.mark.parametrize("at", ["first", "last"])
@pytest.mark.parametrize("mean", [3, 90])
def test_loss_and_gradient_of_a_reduced_hub(gpu_lib, oracle_mod, K, S, at, mean):
    """A reduced graph with rows of a few thousand entries: loss and gradient
    within the bars of the loss parity test, 1e-4 relative."""
    gr = gpu_lib
    n = 6000
    g = _hubs(n, mean, 1, 5000, 7, at)
    agg = (np.arange(n) // 2).astype(np.int32)
    nc = n // 2
    uc, vc, wc = oracle_mod.coarsen(n, g.u, g.v, g.w, agg, nc)
    wc = wc.astype(np.float32).astype(np.float64)
    X = oracle_mod.smooth(n, g.u, g.v, g.w, K, 2).astype(np.float32)
    L_ref, g_ref, _, _ = oracle_mod.loss(n, g.u, g.v, g.w, nc, uc, vc, wc, agg, X.astype(np.float64), S)
    F = gr.graph_reduce_create(n, g.u, g.v, g.w)
    C = gr.graph_reduce_coarsen(F, torch.from_numpy(agg).to(DEV), nc)
    w = torch.from_numpy(wc).float().to(DEV)
    loss, saved = gr.graph_reduce_loss_fwd(F, C, torch.from_numpy(agg).to(DEV), torch.from_numpy(X).to(DEV), w, S)
    grad = gr.graph_reduce_loss_bwd(C, saved, K, w, S, 0.7, torch.ones(1, device=DEV)).double().cpu().numpy()
    assert abs(loss.item() - L_ref) <= 1e-4 * abs(L_ref) + 1e-7
    assert np.linalg.norm(grad - g_ref) <= 1e-4 * np.linalg.norm(g_ref)


@pytest.mark.parametrize("k,normalized", [(1, False), (5, True), (8, False), (32, True)])
@pytest.mark.parametrize("hub_deg,mean,at", [(64, 1, "first"), (65, 1, "first"), (15000, 6, "first"), (15000, 90, "last")])
def test_rayleigh_quotients(gpu_lib, k, normalized, hub_deg, mean, at):
    """x' L x / x' B x of the returned columns, FP64 in another order of the
    sums: 1e-11 relative (2 x 10^5 nodes or a million edges at 2^-53 each)."""
    gr = gpu_lib
    n = 20000
    g = _hubs(n, mean, 2, hub_deg, 11, at)
    levels = [gr.graph_reduce_create(n, g.u, g.v, g.w)]
    for r in (10, 10):
        q = levels[-1].n
        agg = torch.from_numpy((np.arange(q) // r).astype(np.int32)).to(DEV)
        levels.append(gr.graph_reduce_coarsen(levels[-1], agg, -(-q // r)))
    U, lam, rq = gr.graph_reduce_eigensolve(levels, k, normalized=normalized, galerkin_mass=True, iters=3)
    u, v, w = (torch.from_numpy(x).to(DEV) for x in (g.u, g.v, g.w))
    u, v = u.long(), v.long()
    num = (w[:, None] * (U[u] - U[v]) ** 2).sum(0)
    B = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, u, w).index_add_(0, v, w)
    den = ((B[:, None] if normalized else 1.0) * U * U).sum(0)
    want = (num / den).cpu().numpy()
    assert np.all(np.isfinite(want)) and np.abs(rq / want - 1).max() <= 1e-11


@pytest.mark.parametrize("hub_deg,mean,at", [(125, 1, "first"), (128, 1, "last"), (129, 1, "first"), (8000, 4, "first"),
                                             (8000, 30, "last"), (8000, 40, "first")])
def test_colouring(gpu_lib, oracle_mod, hub_deg, mean, at):
    """Rows on both sides of the length that a thread walks, bit for bit."""
    gr = gpu_lib
    n = 9000
    g = _hubs(n, mean, 3, hub_deg, 13, at)
    G = gr.graph_reduce_create(n, g.u, g.v, g.w)
    for seed in (0, 5):
        col, nc = gr.graph_reduce_colour(G, seed)
        ref, rnc = oracle_mod.colour(n, g.u, g.v, seed)
        assert nc == rnc and np.array_equal(col.cpu().numpy(), ref)


def test_colouring_of_many_leaves(gpu_lib, oracle_mod):
    """A star: more leaves become ready at once than a block lists in shared memory."""
    gr = gpu_lib
    n = 100000
    u, v = np.full(n - 1, 777, np.int32), np.setdiff1d(np.arange(n, dtype=np.int32), [777])
    u, v, w = W.canonicalize(n, u, v, np.ones(n - 1))
    G = gr.graph_reduce_create(n, u, v, w)
    for seed in (0, 5, 6):
        col, nc = gr.graph_reduce_colour(G, seed)
        ref, rnc = oracle_mod.colour(n, u, v, seed)
        assert nc == rnc and np.array_equal(col.cpu().numpy(), ref)


@pytest.mark.parametrize("hub_deg", [2100, 8000])
@pytest.mark.parametrize("at", ["first", "last"])
def test_csr_rows(gpu_lib, oracle_mod, hub_deg, at):
    """Degrees and row weights of hubs on a sparse graph, seen through FP64
    sweeps: 1e-12, the bar of the smoothing parity tests."""
    gr = gpu_lib
    n, K, S = 9001, 8, 3
    g = _hubs(n, 4, 2, hub_deg, 17, at)
    G = gr.graph_reduce_create(n, g.u, g.v, g.w)
    X = torch.empty(n, K, dtype=torch.float64, device=DEV)
    gr.graph_reduce_smooth(G, X, S)
    ref = oracle_mod.smooth(n, g.u, g.v, g.w, K, S)
    assert (np.linalg.norm(X.cpu().numpy() - ref, axis=0) / np.linalg.norm(ref, axis=0)).max() <= 1e-12
    agg = torch.from_numpy((np.arange(n) // 3).astype(np.int32)).to(DEV)
    u, v, w = gr.graph_reduce_get_edges(gr.graph_reduce_coarsen(G, agg, -(-n // 3)), on_host=True)
    ur, vr, wr = oracle_mod.coarsen(n, g.u, g.v, g.w, agg.cpu().numpy(), -(-n // 3))
    assert np.array_equal(u.numpy(), ur) and np.array_equal(v.numpy(), vr) and np.array_equal(w.numpy(), wr)
