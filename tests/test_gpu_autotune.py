"""The tuner's probe runs of the models with three and four compartments: the tuned options
give the oracle's results."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T_probe", [1, 100])
@pytest.mark.parametrize("model", [O.SIR, O.SEIR, O.SWIR])
def test_tuned_run_equals_the_oracle(cuda_lib, model, T_probe):
    f = cuda_lib
    g = W.rmat(10, 8, seed=401)
    seeds = W.seed_set(g.n, 20, seed=402)
    graph = f.Graph(g.row_ptr, g.col_idx)
    opts = f.fsgp_options()
    prm = dict(beta=0.05, gamma=0.1, alpha=0.4, mu=0.05, nu=0.3)
    f.fsgp_autotune(graph.handle, model, f.fsgp_params(ic_mode=0, ic_p=0.0, **prm), seeds, len(seeds), 40, T_probe, 9, opts)
    out = f.simulate(graph, model, [seeds], 40, 12, 9, options=opts, **prm)
    ref = O.simulate(model, g.row_ptr, g.col_idx, seeds, R=40, T=12, rng_seed=9, **prm)
    assert np.array_equal(out["counts"][0].cpu().numpy().astype(np.uint64), ref.counts)
    assert np.array_equal(out["freq"][0].cpu().numpy().view(np.uint32), ref.freq)
    graph.close()
