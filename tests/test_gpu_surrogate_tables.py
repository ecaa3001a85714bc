"""The surrogate's long-row tables, built on the graph's first use: no long rows, long rows of
one direction only, every row long (mean degree above a quarter of the bound), chunk
remainders, and rows without arcs.  Tolerances as in test_gpu_surrogate; the two calls add
in different orders at most (float32 sums of at most 3,000 terms)."""
import numpy as np
import pytest

import workloads as W
from oracle import surrogate_ref as S
from tests.test_gpu_surrogate import _check_forward, _check_grad

pytestmark = pytest.mark.gpu


def _graph(kind, n):
    rng = np.random.default_rng(n)
    d = rng.integers(0, 8, size=n)
    p = None
    if kind == "in_long":
        d[[0, 7, n - 1]] = [31, 32, 1025]
    elif kind == "out_long":
        p = np.r_[[0.2, 0.1, 0.004], np.full(n - 3, 0.696 / (n - 3))]
    elif kind == "dense":
        d = rng.integers(64, 130, size=n)
    elif kind == "one_sided":      # every arc into or out of a few nodes
        d[:] = 0
        d[5] = n
        d[100:] = 1
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    col = rng.choice(n, size=int(row_ptr[-1]), p=p).astype(np.int32)
    return W.Graph(row_ptr, col, kind)


@pytest.mark.parametrize("kind", ["none", "in_long", "out_long", "dense", "one_sided"])
def test_first_and_second_call(cuda_lib, kind):
    import torch
    n = 2500
    g = _graph(kind, n)
    graph = cuda_lib.Graph(g.row_ptr, g.col_idx)
    sg = cuda_lib.Surrogate(3)
    theta = S.init_params(4).astype(np.float32)
    sg.set_params(theta)
    seeds = np.arange(0, n, 90, dtype=np.int32)
    x = S.features(g.row_ptr, g.col_idx, seeds, 0.05, 0.1)
    y = np.random.default_rng(5).random(n).astype(np.float32)
    yd = torch.from_numpy(y).cuda()
    loss, grad = sg.grad(graph, seeds, 0.05, 0.1, yd)
    _check_grad(loss, grad, theta, g, x, y)
    _check_forward(sg.forward(graph, seeds, 0.05, 0.1).cpu().numpy(), theta, g, x)
    _, again = sg.grad(graph, seeds, 0.05, 0.1, yd)
    assert np.linalg.norm(grad - again) <= 1e-3 * np.linalg.norm(grad)
    # a graph whose first call screens
    other = cuda_lib.Graph(g.row_ptr, g.col_idx)
    cands = np.random.default_rng(7).integers(0, n, size=(3, 4)).astype(np.int32)
    first = sg.screen(other, cands, 0.02, 0.1)
    want = np.array([float(sg.forward(graph, c, 0.02, 0.1).sum()) for c in cands])
    assert np.allclose(first, want, rtol=1e-3)
