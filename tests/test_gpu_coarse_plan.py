"""The automatic sweep kernel of a coarse graph does not depend on how it was
assembled: row by row, or by a global sort (an aggregate of more than 1,024
slots).  Rows known to be short count on created graphs only."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("clique", [False, True])
def test_plan_of_a_sparse_coarse_graph(gpu_lib, clique):
    gr = gpu_lib
    nc, size, band = 16000, 36, 10  # coarse rows of 20; an aggregate's clique has 36 x 35 slots
    A = np.repeat(np.arange(nc), band)
    B = A + np.tile(np.arange(1, band + 1), nc)
    a, b = size * A[B < nc], size * B[B < nc] + 1
    i, j = np.triu_indices(size, 1) if clique else (np.zeros(size - 1, int), np.arange(1, size))
    a = np.concatenate([a, (size * np.arange(nc)[:, None] + i).ravel()])
    b = np.concatenate([b, (size * np.arange(nc)[:, None] + j).ravel()])
    n = nc * size
    G = gr.graph_reduce_create(n, *W.canonicalize(n, a, b, np.ones(a.size)))
    agg = torch.from_numpy((np.arange(n) // size).astype(np.int32)).to(DEV)
    C = gr.graph_reduce_coarsen(G, agg, nc)
    u, v, w = gr.graph_reduce_get_edges(C)
    assert C.m == int((B < nc).sum())
    for dt in (torch.float64, torch.bfloat16, torch.float32):
        assert gr.graph_reduce_sweep_plan(C, 8, dt) == gr.GR_SWEEP_STREAM
    created = gr.graph_reduce_create(nc, u, v, w)
    assert gr.graph_reduce_sweep_plan(created, 8, torch.float64) != gr.GR_SWEEP_STREAM
