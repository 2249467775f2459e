"""Member lists of a node map around the sizes where their sorting changes
(registers up to 128 members, shared memory up to 1,024, a radix sort above):
the reduced data set, which adds the members in ascending id, against the
oracle bit for bit, with zeros and FP32 subnormal numbers among the data."""
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


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("d,sizes", [(1, [1, 32, 33, 64, 65, 128, 129]), (7, [1024, 1023]), (16, [1025])])
def test_member_sums(gr, oracle_mod, dtype, d, sizes):
    g = W.random_sparse(4003, 9000, seed=d)
    rest = g.n - sum(sizes)
    agg = np.concatenate([np.full(s, i) for i, s in enumerate(sizes)] + [len(sizes) + np.arange(rest) % 40])
    rng = np.random.default_rng(7)
    agg, nc = rng.permutation(agg).astype(np.int32), len(sizes) + 40
    F = rng.normal(size=(g.n, d)).astype(dtype)
    F[::97] = 0.0
    F[5::101] *= 1e-42
    G = gr.graph_reduce_create(g.n, g.u, g.v, g.w)
    C = gr.graph_reduce_coarsen(G, torch.from_numpy(agg).to(DEV), nc)
    for mean in (False, True):
        out = gr.graph_reduce_reduce_data([C], torch.from_numpy(F).to(DEV), mean=mean).cpu().numpy()
        assert np.array_equal(out, oracle_mod.reduce_features(agg, nc, F, mean).astype(dtype))
