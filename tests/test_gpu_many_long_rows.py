"""Small graphs with more rows of 256 in-arcs than there are resident warps, most rows being
short: the step's CTAs go by work, in the persistent loop and in a launch per step."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [64, 1000])
@pytest.mark.parametrize("options", [{}, {"persistent": -1}])
def test_many_long_rows(cuda_lib, options, R):
    import torch
    rng = np.random.default_rng(51)
    n, n_long = 16_000, 4_000
    d = rng.integers(0, 6, size=n)
    d[:n_long] = rng.integers(256, 300, size=n_long)
    d = d[rng.permutation(n)]
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    g = W.Graph(row_ptr, rng.integers(0, n, size=int(row_ptr[-1])).astype(np.int32), "many long rows")
    seeds = W.seed_set(n, 200, seed=52)
    graph = cuda_lib.Graph(g.row_ptr, g.col_idx)
    prm = dict(beta=0.02, gamma=0.2, alpha=0.4, mu=0.1, nu=0.5)
    for model in (O.SIS, O.LT, O.SWIR, O.IC):
        out = cuda_lib.simulate(graph, model, [seeds], R, 3, 53, options=dict(options), **prm)
        torch.cuda.synchronize()
        ref = O.simulate(model, g.row_ptr, g.col_idx, seeds, R=R, T=3, rng_seed=53, **prm)
        assert np.array_equal(out["counts"][0].cpu().numpy().astype(np.uint64), ref.counts), model
        assert np.array_equal(out["freq"][0].cpu().numpy().view(np.uint32), ref.freq), model
    graph.close()
