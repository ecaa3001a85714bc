"""The surrogate's fused layers at sizes around their 128-row tiles, with rows of no arcs,
around the eight-arc rounds and above the split of long rows; screening with few seeds
(one cluster launch per candidate) and with many.  Tolerances as in test_gpu_surrogate."""
import numpy as np
import pytest

import workloads as W
from oracle import surrogate_ref as S
from tests.test_gpu_surrogate import _check_forward, _check_grad

pytestmark = pytest.mark.gpu


def _graph(n, seed):
    rng = np.random.default_rng(seed)
    d = rng.choice([0, 1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 40], size=n)
    d[:min(n, 6)] = [31, 32, 33, 255, 256, 700][:min(n, 6)]
    d = d[rng.permutation(n)]
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    return W.Graph(row_ptr, rng.integers(0, n, size=int(row_ptr[-1])).astype(np.int32), "tiles")


@pytest.mark.parametrize("n", [1, 127, 128, 129, 1000])
def test_forward_around_a_tile(cuda_lib, n):
    g = _graph(n, 50 + n)
    graph = cuda_lib.Graph(g.row_ptr, g.col_idx)
    sg = cuda_lib.Surrogate(3)
    theta = S.init_params(4).astype(np.float32)
    sg.set_params(theta)
    seeds = np.arange(0, n, 9, dtype=np.int32)
    x = S.features(g.row_ptr, g.col_idx, seeds, 0.05, 0.1)
    _check_forward(sg.forward(graph, seeds, 0.05, 0.1).cpu().numpy(), theta, g, x)


@pytest.mark.parametrize("n", [2431, 2432, 2433, 2465])
def test_gradient_with_a_ragged_last_tile(cuda_lib, n):
    """(At the size of the gradient bounds' own tests: a bound per block is a norm over many
    rows, which a single ReLU taking the other side in bfloat16 must not dominate.)"""
    import torch
    g = _graph(n, 50 + n)
    graph = cuda_lib.Graph(g.row_ptr, g.col_idx)
    sg = cuda_lib.Surrogate(3)
    theta = S.init_params(4).astype(np.float32)
    sg.set_params(theta)
    seeds = np.arange(0, n, 90, dtype=np.int32)
    x = S.features(g.row_ptr, g.col_idx, seeds, 0.05, 0.1)
    y = np.random.default_rng(5).random(n).astype(np.float32)
    loss, grad = sg.grad(graph, seeds, 0.05, 0.1, torch.from_numpy(y).cuda())
    _check_grad(loss, grad, theta, g, x, y)


@pytest.mark.parametrize("k", [1, 64, 65])
def test_screening_restores_features(cuda_lib, k):
    g = _graph(1000, 61)
    graph = cuda_lib.Graph(g.row_ptr, g.col_idx)
    sg = cuda_lib.Surrogate(6)
    cands = np.random.default_rng(7).integers(0, g.n, size=(9, k)).astype(np.int32)
    cands[4] = cands[3][0]   # one node repeated
    first = sg.screen(graph, cands, 0.02, 0.1)
    again = sg.screen(graph, cands[::-1].copy(), 0.02, 0.1)[::-1]
    want = np.array([float(sg.forward(graph, c, 0.02, 0.1).sum()) for c in cands])
    # float32 sums of at most 1000 terms in any order: 1000 * 2^-24 relative
    assert np.allclose(first, want, rtol=1e-4) and np.allclose(again, want, rtol=1e-4)
