"""Per-realization counts of wide runs, whose counters take shared memory beside the row
kernels' tiles: the degree-class and the fused kernels, launched and captured."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("options", [{}, {"fuse_rows": -1}, {"fuse_rows": -1, "capture_graph": 1}, {"capture_graph": 1}])
@pytest.mark.parametrize("model", [O.SIR, O.SWIR, O.IC, O.SEIR])
def test_per_realization_counts(cuda_lib, model, options):
    import torch
    g = W.ba(1500, 6, seed=61)
    seeds = W.seed_set(g.n, 40, seed=62)
    graph = cuda_lib.Graph(g.row_ptr, g.col_idx)
    prm = dict(beta=0.05, gamma=0.2, alpha=0.4, mu=0.1, nu=0.5)
    R, T = 1021, 4
    for run in range(2):   # with counters, without, and with them again
        out = cuda_lib.simulate(graph, model, [seeds], R, T, 63, per_real=True, options=dict(options), **prm)
        plain = cuda_lib.simulate(graph, model, [seeds], R, T, 63, options=dict(options), **prm)
        torch.cuda.synchronize()
        ref = O.simulate(model, g.row_ptr, g.col_idx, seeds, R=R, T=T, rng_seed=63, **prm)
        assert np.array_equal(out["per_real"][0].cpu().numpy().view(np.uint32), ref.per_real), run
        assert np.array_equal(plain["counts"][0].cpu().numpy().astype(np.uint64), ref.counts), run
    graph.close()
