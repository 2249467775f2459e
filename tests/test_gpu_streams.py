"""Calls that return before their work is done, on streams other than the
default one: a refused call has left the stream idle, results and the lifetime
of the tensors passed are those of a call that waited.  Results are compared
bit for bit with the same call on the default stream (fixed order of every
sum)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _graph(n, deg, seed):
    g = W.random_sparse(n, deg * n, seed=seed)
    return g, torch.from_numpy((np.arange(n) // 8).astype(np.int32)).to(DEV), -(-n // 8)


@pytest.mark.parametrize("call", ["loss", "scale"])
def test_refused_label_leaves_the_stream_idle(gpu_lib, call):
    gr = gpu_lib
    n, K = 400000, 32  # the fine pass takes some 100 us after the labels are known to be bad
    g, agg, nc = _graph(n, 8, 1)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        F = gr.graph_reduce_create(n, g.u, g.v, g.w)
        C = gr.graph_reduce_coarsen(F, agg, nc)
        w = gr.graph_reduce_get_edges(C)[2].float()
        X = torch.ones(n, K, device=DEV)
        bad = agg.clone()
        bad[17] = nc
        side.synchronize()
        with pytest.raises(gr.GraphReduceError) as ei:
            if call == "loss":
                gr.graph_reduce_loss_fwd(F, C, bad, X, w, 2)
            else:
                gr.graph_reduce_scale_edges(F, C, bad, X, w, 2)
        assert side.query()
    assert ei.value.status == 1
