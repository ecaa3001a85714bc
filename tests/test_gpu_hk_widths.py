"""Hegselmann-Krause at every lane-team width of the step kernel (8, 16 and 32 lanes per
node, one to three segments per row), with node counts off the transposes' 32 x 32 tiles
and rows of 0, 1, 7, 8, 9 and several hundred in-arcs, equals the oracle bit for bit."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 1003])
@pytest.mark.parametrize("R", [1, 32, 40, 64, 65, 96, 128, 200, 256])
def test_widths(cuda_lib, R, n):
    import torch
    rng = np.random.default_rng(100 * R + n)
    d = rng.choice([0, 1, 2, 7, 8, 9, 16, 17], size=n)
    d[0] = 400
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    col = rng.integers(0, n, size=int(row_ptr[-1])).astype(np.int32)
    h0 = rng.uniform(-1, 1, size=(R, n)).astype(np.float32)
    graph = cuda_lib.Graph(row_ptr, col)
    want, changes = O.hk(row_ptr, col, h0, T=6, eps=0.4)
    h, ch = cuda_lib.hk(graph, h0, 6, 0.4)
    assert np.array_equal(h.view(np.uint32), want.view(np.uint32))
    assert np.array_equal(ch.astype(np.uint64), changes)
    h, ch = cuda_lib.hk(graph, torch.from_numpy(h0).cuda(), 6, 0.4)
    assert np.array_equal(h.cpu().numpy().view(np.uint32), want.view(np.uint32))
    assert np.array_equal(ch.cpu().numpy().astype(np.uint64), changes)
    bad = torch.from_numpy(h0).cuda()
    bad[R - 1, n - 1] = float("nan")
    with pytest.raises(cuda_lib.FsgpError):
        cuda_lib.hk(graph, bad, 1, 0.4)


@pytest.mark.parametrize("longest", [17, 31, 32, 33, 65, 255])
@pytest.mark.parametrize("R", [32, 64, 128])
def test_long_rows(cuda_lib, R, longest):
    # rows on both sides of the bound for a CTA of their own, and graphs without such rows
    n = 700
    rng = np.random.default_rng(longest * R)
    d = rng.choice([0, 1, 2, 7], size=n)
    d[[3, 350, n - 1]] = longest
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    col = rng.integers(0, n, size=int(row_ptr[-1])).astype(np.int32)
    h0 = rng.uniform(-1, 1, size=(R, n)).astype(np.float32)
    want, changes = O.hk(row_ptr, col, h0, T=4, eps=0.4)
    h, ch = cuda_lib.hk(cuda_lib.Graph(row_ptr, col), h0, 4, 0.4)
    assert np.array_equal(h.view(np.uint32), want.view(np.uint32))
    assert np.array_equal(ch.astype(np.uint64), changes)
