"""FP32 affinities of 32 columns, whose rows a warp reads together: edge counts
around a warp and a block, and a graph whose edges end anywhere.  Compared with
the FP64 definition on the same FP32 block, within 1e-5 as every FP32 affinity."""
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


@pytest.mark.parametrize("g", [W.path(2), W.path(32), W.path(33), W.path(34), W.path(258),
                               W.random_sparse(3001, 20011, seed=5)], ids=lambda g: "m%d" % g.m)
def test_affinity_of_32_columns(gr, oracle_mod, g):
    X = torch.from_numpy(np.random.default_rng(g.m).standard_normal((g.n, 32))).to(DEV).float()
    G = gr.graph_reduce_create(g.n, g.u, g.v, g.w)
    d, a = (torch.full((g.m,), -1.0, dtype=torch.float32, device=DEV) for _ in range(2))
    gr.graph_reduce_affinity(G, X, d, a)
    dref, aref = oracle_mod.affinity(g.n, g.u, g.v, X.double().cpu().numpy(), want_a=True)
    assert np.abs(d.cpu().numpy() - dref).max() <= 1e-5 and np.abs(a.cpu().numpy() - aref).max() <= 1e-5
