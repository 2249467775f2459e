"""A refused aggregation writes no label: the last pass merges and labels on the
device before the host has seen the error flags and the proposal counts."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("passes", [1, 2])  # with two, the first pass's counts are looked at after the second
@pytest.mark.parametrize("why,status", [("negative", 1), ("nan", 1), ("budget", 4)])
def test_labels_stay(gpu_lib, dtype, passes, why, status):
    gr = gpu_lib
    g = W.grid2d(40, 30)
    G = gr.graph_reduce_create(g.n, g.u, g.v, g.w)
    d = torch.from_numpy(np.random.default_rng(1).uniform(0.1, 1.0, g.m)).to(DEV, dtype)
    target = g.n // 4
    agg = torch.full((g.n,), -7, dtype=torch.int32, device=DEV)
    if why == "negative":
        d[g.m // 2] = -0.5
    elif why == "nan":
        d[g.m // 2] = float("nan")
    with pytest.raises(gr.GraphReduceError) as ei:
        gr.graph_reduce_aggregate(G, d, target, passes, max_proposals=3 if why == "budget" else 0, agg_out=agg)
    assert ei.value.status == status
    torch.cuda.synchronize()
    assert torch.equal(agg, torch.full_like(agg, -7))
    # the same call on sound input writes every label
    d = d.abs().nan_to_num(0.5)
    nc = gr.graph_reduce_aggregate(G, d, target, passes, agg_out=agg)[1]
    assert int(agg.min()) == 0 and int(agg.max()) == nc - 1
