"""Branches of the loss and its adjoint: every vector width,
no sweep, short and long reduced rows, small and large groups, and blocks that
start off a 16-byte boundary.  Bars: those of the loss parity test (1e-4
relative on the loss and on the gradient's norm; FP32 vectors of at most a few
thousand rows, sums in FP64 from the warp level up)."""
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


def _groups(n, sizes, seed):
    """A map of n nodes onto labels with the given sizes, the rest spread evenly over 40 more."""
    rng = np.random.default_rng(seed)
    lab = np.concatenate([np.full(s, i) for i, s in enumerate(sizes)])
    rest = n - lab.size
    lab = np.concatenate([lab, len(sizes) + np.arange(rest) % 40]).astype(np.int32)
    return rng.permutation(lab), len(sizes) + 40


def _offset(t, off):
    """The same values in a block that starts `off` floats past an aligned address."""
    buf = torch.empty(t.numel() + 4, dtype=t.dtype, device=t.device)
    view = buf[off:off + t.numel()].view(t.shape)
    view.copy_(t)
    return view


CASES = [(4, 2, 3, [1, 32, 33], 0), (8, 0, 3, [1, 2], 0), (16, 1, 3, [64, 65], 1), (24, 3, 3, [1024], 0),
         (24, 2, 20, [1025, 7], 3), (32, 5, 20, [300], 0)]


@pytest.mark.parametrize("K,S,deg,sizes,off", CASES)
def test_loss_paths(gr, oracle_mod, K, S, deg, sizes, off):
    g = W.random_sparse(3001, deg * 3001, seed=K + S)
    agg, nc = _groups(g.n, sizes, 5)
    uc, vc, wc = oracle_mod.coarsen(g.n, g.u, g.v, g.w, agg, nc)
    wc = wc.astype(np.float32).astype(np.float64)
    X = oracle_mod.smooth(g.n, g.u, g.v, g.w, K, 2).astype(np.float32)
    L_ref, g_ref, _, _ = oracle_mod.loss(g.n, g.u, g.v, g.w, nc, uc, vc, wc, agg, X.astype(np.float64), S)
    F = gr.graph_reduce_create(g.n, g.u, g.v, g.w)
    C = gr.graph_reduce_create(nc, uc, vc, wc)
    Xd = _offset(torch.from_numpy(X).to(DEV), off)
    w = torch.from_numpy(wc).float().to(DEV)
    saved = _offset(torch.empty(nc * (K + 1) + K, device=DEV), off)
    loss, saved = gr.graph_reduce_loss_fwd(F, C, torch.from_numpy(agg).to(DEV), Xd, w, S, saved=saved)
    grad = gr.graph_reduce_loss_bwd(C, saved, K, w, S, 0.7, torch.ones(1, device=DEV)).double().cpu().numpy()
    assert abs(loss.item() - L_ref) <= 1e-4 * abs(L_ref) + 1e-7
    assert np.linalg.norm(grad - g_ref) <= 1e-4 * np.linalg.norm(g_ref)


def test_loss_rejects_bad_labels(gr, oracle_mod):
    g = W.random_sparse(500, 1500, seed=2)
    agg, nc = _groups(g.n, [3], 6)
    uc, vc, wc = oracle_mod.coarsen(g.n, g.u, g.v, g.w, agg, nc)
    F = gr.graph_reduce_create(g.n, g.u, g.v, g.w)
    C = gr.graph_reduce_create(nc, uc, vc, wc)
    agg = agg.copy()
    agg[17] = nc
    with pytest.raises(gr.GraphReduceError) as ei:
        gr.graph_reduce_loss_fwd(F, C, torch.from_numpy(agg).to(DEV), torch.ones(g.n, 4, device=DEV),
                                 torch.from_numpy(wc).float().to(DEV), 1)
    assert ei.value.status == 1
