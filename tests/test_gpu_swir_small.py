"""SWIR on small graphs: the persistent loop's shape follows from the longest row and the
width (two teams per row below 64 in-arcs and up to two words, 8-bit counters below 256)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("longest", [9, 63, 64, 255, 256])
@pytest.mark.parametrize("R,n_sets", [(20, 1), (64, 1), (33, 3), (300, 1)])
def test_longest_row(cuda_lib, R, n_sets, longest):
    rng = np.random.default_rng(71)
    n = 700
    d = rng.integers(0, 10, size=n)
    d[[0, 250, 699]] = longest
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    g = W.Graph(row_ptr, rng.integers(0, n, size=int(row_ptr[-1])).astype(np.int32), "longest")
    sets = [W.seed_set(n, 60, seed=72 + i) for i in range(n_sets)]
    prm = dict(beta=0.1, gamma=0.2, mu=0.1, nu=0.5)
    graph = cuda_lib.Graph(g.row_ptr, g.col_idx)
    for options in ({}, {"persistent": -1}):
        out = cuda_lib.simulate(graph, O.SWIR, sets, R, 6, 73, options=dict(options), **prm)
        for i, seeds in enumerate(sets):
            ref = O.simulate(O.SWIR, g.row_ptr, g.col_idx, seeds, R=R, T=6, rng_seed=73, **prm)
            assert np.array_equal(out["counts"][i].cpu().numpy().astype(np.uint64), ref.counts), options
            assert np.array_equal(out["freq"][i].cpu().numpy().view(np.uint32), ref.freq), options
    graph.close()
