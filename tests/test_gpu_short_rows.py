"""The automatic sweep kernel on graphs with long mean rows: FP64 and BF16
blocks take the row-group kernel when no row has more than 64 slots on a side
of the diagonal, the streaming kernel as soon as one has, whichever side it is
on; FP32 blocks keep the streaming kernel.  The forced kernels are compared
with the oracle elsewhere; here the automatic one, FP64 within 1e-12."""
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


@pytest.mark.parametrize("side,length,short", [("upper", 64, True), ("upper", 65, False), ("lower", 64, True),
                                               ("lower", 65, False)])
def test_row_length_border(gr, oracle_mod, side, length, short):
    n, band = 2000, 20  # a band of 20 neighbours on each side, and one hub at an end
    a = np.repeat(np.arange(n), band)
    b = a + np.tile(np.arange(1, band + 1), n)
    hub = np.full(length - band, 0 if side == "upper" else n - 1)
    far = np.arange(200, 200 + length - band)
    a, b = np.concatenate([a[b < n], hub]), np.concatenate([b[b < n], far])
    rng = np.random.default_rng(length)
    u, v, w = W.canonicalize(n, a, b, rng.uniform(0.1, 2.0, a.size))
    G = gr.graph_reduce_create(n, u, v, w)
    K, S = 8, 3
    plan = {dt: gr.graph_reduce_sweep_plan(G, K, dt) for dt in (torch.float64, torch.float32, torch.bfloat16)}
    want = gr.GR_SWEEP_ROW if short else gr.GR_SWEEP_STREAM
    assert plan[torch.float64] == plan[torch.bfloat16] == want and plan[torch.float32] == gr.GR_SWEEP_STREAM
    X = torch.empty(n, K, dtype=torch.float64, device=DEV)
    gr.graph_reduce_smooth(G, X, S)
    ref = oracle_mod.smooth(n, u, v, w, K, S)
    err = np.linalg.norm(X.cpu().numpy() - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() <= 1e-12
