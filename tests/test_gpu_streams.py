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


def _loss_and_data(gr, F, C, agg, X, w):
    loss, saved = gr.graph_reduce_loss_fwd(F, C, agg, X, w, 2)
    return loss, saved, gr.graph_reduce_reduce_data([C], X)


def _equal(got, want):
    return all(torch.equal(a, b) for a, b in zip(got, want))


def test_caller_on_another_stream(gpu_lib, monkeypatch):
    """Graphs of the default stream and of a side stream, each called from the
    other: the results are there, and the graph's stream is idle, on return;
    other streams are not waited for."""
    gr = gpu_lib
    n, K = 200000, 16
    g, agg, nc = _graph(n, 6, 2)
    X = torch.randn(n, K, device=DEV, generator=torch.Generator(device=DEV).manual_seed(3))
    home, side = torch.cuda.current_stream(), torch.cuda.Stream()
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: pytest.fail("the whole device was waited for"))
    want = None
    for owner, caller in ((home, home), (home, side), (side, home)):
        with torch.cuda.stream(owner):
            F = gr.graph_reduce_create(n, g.u, g.v, g.w)
            C = gr.graph_reduce_coarsen(F, agg, nc)
            w = gr.graph_reduce_get_edges(C)[2].float()
        owner.synchronize()
        with torch.cuda.stream(caller):
            got = _loss_and_data(gr, F, C, agg, X, w)
            if owner != caller:
                assert owner.query()
        caller.synchronize()
        want = want or got
        assert _equal(got, want)


def test_tensor_of_a_third_stream(gpu_lib):
    """A block allocated on another stream than the graph's and freed right
    after the call is not handed out while the call still reads it."""
    gr = gpu_lib
    n, K = 400000, 32
    g, agg, nc = _graph(n, 8, 4)
    X = torch.randn(n, K, device=DEV, generator=torch.Generator(device=DEV).manual_seed(5))
    F = gr.graph_reduce_create(n, g.u, g.v, g.w)
    C = gr.graph_reduce_coarsen(F, agg, nc)
    w = gr.graph_reduce_get_edges(C)[2].float()
    want = _loss_and_data(gr, F, C, agg, X, w)
    side = torch.cuda.Stream()
    for _ in range(5):
        for i in range(2):
            with torch.cuda.stream(side):
                Y = X.clone()
            side.synchronize()
            got = gr.graph_reduce_loss_fwd(F, C, agg, Y, w, 2) if i == 0 else (gr.graph_reduce_reduce_data([C], Y),)
            del Y
            with torch.cuda.stream(side):
                Z = torch.full_like(X, float("nan"))
            torch.cuda.synchronize()
            del Z
            assert _equal(got, want[:2] if i == 0 else want[2:])
