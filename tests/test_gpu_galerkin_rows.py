"""Row classes of the Galerkin product around their borders (32, 128 and 1,024
slots a row, the global sort past that), many fine edges between two
aggregates and members without edges, against the oracle: pattern and weights
bit for bit, degrees through one smoothing sweep (FP64, 1e-12)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def gr():
    from paper_1812_08942_gb300 import build as B
    B.build()
    import paper_1812_08942_gb300 as gr
    gr.load()
    return gr


def _check(gr, oracle_mod, g, agg, nc):
    uc, vc, wc = oracle_mod.coarsen(g.n, g.u, g.v, g.w, agg, nc)
    G = gr.graph_reduce_create(g.n, g.u, g.v, g.w)
    C = gr.graph_reduce_coarsen(G, torch.from_numpy(agg).to(DEV), nc)
    cu, cv, cw = (t.numpy() for t in gr.graph_reduce_get_edges(C, on_host=True))
    assert np.array_equal(cu, uc) and np.array_equal(cv, vc) and np.array_equal(cw, wc)
    ref = oracle_mod.smooth(nc, uc, vc, wc, 4, 1)
    X = torch.empty(nc, 4, dtype=torch.float64, device=DEV)
    gr.graph_reduce_smooth(C, X, 1)
    err = np.linalg.norm(X.cpu().numpy() - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() <= 1e-12


def _star(leaves, extra, seed):
    """A hub with `leaves` leaves (its row has that many slots) and a random rest."""
    n = 1 + leaves + extra
    rng = np.random.default_rng(seed)
    a = np.concatenate([np.zeros(leaves, np.int64), rng.integers(1, n, 3 * n)])
    b = np.concatenate([np.arange(1, leaves + 1), rng.integers(1, n, 3 * n)])
    u, v, w = W.canonicalize(n, a, b, rng.uniform(0.1, 2.0, a.size))
    return W.Graph(n, u, v, w)


@pytest.mark.parametrize("leaves", [31, 32, 33, 128, 129, 1024, 1025, 5000])
def test_hub_row(gr, oracle_mod, leaves):
    g = _star(leaves, 500, leaves)
    agg = np.concatenate([[0], 1 + np.random.default_rng(1).permutation(np.arange(g.n - 1) // 2)]).astype(np.int32)
    _check(gr, oracle_mod, g, agg, int(agg.max()) + 1)


@pytest.mark.parametrize("nodes,groups", [(400, 12), (900, 7), (900, 30), (3000, 12), (3000, 4)])
def test_runs(gr, oracle_mod, nodes, groups):
    # few aggregates of many nodes: long rows, runs of tens to thousands of edges
    g = W.random_sparse(nodes, 12 * nodes, seed=nodes + groups)
    agg = np.random.default_rng(2).permutation(np.arange(nodes) % groups).astype(np.int32)
    _check(gr, oracle_mod, g, agg, groups)


@pytest.mark.parametrize("shape", [(37, 23), (128, 96)])
def test_short_rows(gr, oracle_mod, shape):
    # every row within 32 slots: a thread each
    g = W.grid2d(*shape, weights=lambda m: np.random.default_rng(4).uniform(0.1, 2.0, m))
    ids = np.arange(g.n)
    for agg in (ids // 2, ids // 4, (ids % shape[0]) // 2 + (shape[0] + 1) // 2 * (ids // shape[0] // 4)):
        _check(gr, oracle_mod, g, agg.astype(np.int32), int(agg.max()) + 1)


def test_isolated(gr, oracle_mod):
    # 3,000 isolated nodes share one label, another is used by one of them alone
    g = _star(300, 7_000, 5)
    n = g.n + 3001
    agg = np.arange(n, dtype=np.int32)
    agg[g.n:g.n + 3000] = 7
    agg[-1] = g.n
    _check(gr, oracle_mod, W.Graph(n, g.u, g.v, g.w), agg, g.n + 1)
