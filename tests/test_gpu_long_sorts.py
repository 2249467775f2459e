"""The global sorts around the sizes where they change: tiles of 8,192 pairs,
digits of 8 to 10 bits, one to four passes.  A coarse row past 1,024 slots
sends the Galerkin product to a sort of 2 ceil(log2 nc)-bit keys, and the dense
coarse graphs sort their edges by end node.  Integers and weights (sums in
edge order) are compared exactly, a smoothing run on both graphs within
1e-12."""
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


def _smooth_err(gr, oracle_mod, G, n, u, v, w):
    K, S = 8, 2
    X = torch.empty(n, K, dtype=torch.float64, device=DEV)
    gr.graph_reduce_smooth(G, X, S, 0.7, 3, 0)
    ref = oracle_mod.smooth(n, u, v, w, K, S, 0.7, 3, 0)
    return (np.linalg.norm(X.cpu().numpy() - ref, axis=0) / np.linalg.norm(ref, axis=0)).max()


# nodes, edges exactly, labels: about n / merge (one label takes 1,100 nodes
# where the others would leave no row long enough)
@pytest.mark.parametrize("n,m,merge,hub", [
    (300, 8191, 60, 0), (300, 8192, 60, 0), (300, 8193, 60, 0),   # one tile and its edge; one pass
    (500, 3 * 8192 + 5, 5, 0),                                    # 14-bit keys: two passes of 8
    (1500, 40000, 2, 700),                                        # 20 bits: two passes of 10
    (3000, 60000, 2, 1100),                                       # 22 bits: three passes of 8
    (40000, 700001, 2, 1100),                                     # 30 bits: three passes of 10
    (70000, 1200000, 1, 1100),                                    # 34 bits: four passes of 9
])
def test_long_sorts(gr, oracle_mod, n, m, merge, hub):
    rng = np.random.default_rng(n + m)
    key = np.unique(rng.integers(0, n, int(1.4 * m) + 64) * n + rng.integers(0, n, int(1.4 * m) + 64))
    key = key[key // n < key % n]
    while key.size < m:
        more = rng.integers(0, n, 2 * m) * n + rng.integers(0, n, 2 * m)
        key = np.unique(np.concatenate([key, more[more // n < more % n]]))
    key = np.sort(rng.permutation(key)[:m])
    u, v, w = (key // n).astype(np.int32), (key % n).astype(np.int32), rng.uniform(0.5, 2.0, m)
    lab = np.concatenate([np.zeros(hub, np.int64), (hub > 0) + np.arange(n - hub) // merge])
    nc = int(lab.max()) + 1
    agg = rng.permutation(nc)[lab[rng.permutation(n)]].astype(np.int32)
    G = gr.graph_reduce_create(n, u, v, w)
    C = gr.graph_reduce_coarsen(G, torch.from_numpy(agg).to(DEV), nc)
    uc, vc, wc = oracle_mod.coarsen(n, u, v, w, agg, nc)
    gu, gv, gw = (t.numpy() for t in gr.graph_reduce_get_edges(C, on_host=True))
    assert C.n == nc and np.array_equal(gu, uc) and np.array_equal(gv, vc) and np.array_equal(gw, wc)
    assert _smooth_err(gr, oracle_mod, G, n, u, v, w) <= 1e-12
    assert _smooth_err(gr, oracle_mod, C, nc, uc, vc, wc) <= 1e-12
