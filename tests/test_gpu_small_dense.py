"""Short rows on few of them: FP64 and BF16 blocks take the row-group kernel
only where the graph has rows for every SM, and its eight-slot form agrees with
the oracle (FP64 1e-12) and with the streaming kernel (BF16, both rounding the
same sums: 2^-8 per sweep of a column's norm)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _band(n, half, seed=0):
    a = np.repeat(np.arange(n), half)
    b = a + np.tile(np.arange(1, half + 1), n)
    a, b = a[b < n], b[b < n]
    return W.canonicalize(n, a, b, np.random.default_rng(seed).uniform(0.1, 2.0, a.size))


@pytest.mark.parametrize("n,half,K,row64,row16", [(1000, 50, 8, False, False), (1000, 20, 8, True, True),
                                                  (1000, 20, 4, False, True), (12000, 40, 8, True, False),
                                                  (60000, 60, 16, True, True)])
def test_rows_for_every_sm(gpu_lib, n, half, K, row64, row16):
    gr = gpu_lib
    G = gr.graph_reduce_create(n, *_band(n, half))
    plans = [gr.graph_reduce_sweep_plan(G, K, dt) for dt in (torch.float64, torch.bfloat16, torch.float32)]
    assert [p == gr.GR_SWEEP_STREAM for p in plans] == [not row64, not row16, True]


@pytest.mark.parametrize("n,half", [(31, 15), (1111, 20), (3001, 33), (9973, 24)])
@pytest.mark.parametrize("K", [4, 8, 16, 24, 32])
def test_eight_slots(gpu_lib, oracle_mod, n, half, K):
    gr = gpu_lib
    u, v, w = _band(n, half)
    G = gr.graph_reduce_create(n, u, v, w)
    gr.graph_reduce_set_sweep_kernel(G, gr.GR_SWEEP_ROW)
    S = 3
    X = torch.empty(n, K, dtype=torch.float64, device=DEV)
    gr.graph_reduce_smooth(G, X, S)
    ref = oracle_mod.smooth(n, u, v, w, K, S)
    norm = np.maximum(np.linalg.norm(ref, axis=0), 1e-300)
    assert (np.linalg.norm(X.cpu().numpy() - ref, axis=0) / norm).max() <= 1e-12
    Y = [torch.empty(n, K, dtype=torch.bfloat16, device=DEV) for _ in range(2)]
    gr.graph_reduce_smooth(G, Y[0], S)
    gr.graph_reduce_set_sweep_kernel(G, gr.GR_SWEEP_STREAM)
    gr.graph_reduce_smooth(G, Y[1], S)
    a, b = (y.double().cpu().numpy() for y in Y)
    assert (np.linalg.norm(a - b, axis=0) <= S * 2.0 ** -8 * np.linalg.norm(b, axis=0) + 1e-300).all()
