"""Screening seeds of very different out-degrees (none to several rounds of the cluster's
threads, repeated hubs) against the forward pass of each candidate; float32 sums of 30,000
terms in any order: 30000 * 2^-24 = 1.8e-3 relative."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 33, 63, 64])
def test_hub_and_leaf_seeds(cuda_lib, k):
    rng = np.random.default_rng(k)
    n = 30_000
    # two arcs into each node, from one of three hubs and from a node of the first half
    col = np.stack([rng.choice([0, 11, n - 1], size=n, p=[0.6, 0.3, 0.1]), rng.integers(0, n // 2, size=n)], 1)
    row_ptr = np.arange(0, 2 * n + 1, 2, dtype=np.int32)
    graph = cuda_lib.Graph(row_ptr, col.reshape(-1).astype(np.int32))
    sg = cuda_lib.Surrogate(6)
    cands = rng.integers(0, n, size=(6, k)).astype(np.int32)
    cands[0] = 0                      # one hub k times
    cands[1, :] = n - 2               # no out-arcs
    cands[2, ::2] = 11
    cands[3, -1] = n - 1
    cands[4, :3] = [0, 11, n - 1][:min(k, 3)]
    want = np.array([float(sg.forward(graph, c, 0.02, 0.1).double().sum()) for c in cands])
    for order in (np.arange(6), np.arange(6)[::-1]):
        got = sg.screen(graph, np.ascontiguousarray(cands[order]), 0.02, 0.1)
        assert np.allclose(got, want[order], rtol=2e-3)
    again = np.array([float(sg.forward(graph, c, 0.02, 0.1).double().sum()) for c in cands])
    assert np.array_equal(again, want)   # the features were taken back
