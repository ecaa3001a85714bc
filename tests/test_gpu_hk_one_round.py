"""HK without long rows, on both sides of the size at which all nodes have their teams at
once (narrow teams on small CTAs up to there)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off", [-1, 0, 1])
@pytest.mark.parametrize("R", [20, 64, 128])
def test_bound(cuda_lib, R, off):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = sms * 256 // ((R + 31) // 32) + off
    rng = np.random.default_rng(R + off)
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(rng.choice([0, 1, 7, 8, 9, 17], size=n))
    col = rng.integers(0, n, size=int(row_ptr[-1])).astype(np.int32)
    h0 = rng.uniform(-1, 1, size=(R, n)).astype(np.float32)
    want, changes = O.hk(row_ptr, col, h0, T=3, eps=0.4)
    h, ch = cuda_lib.hk(cuda_lib.Graph(row_ptr, col), h0, 3, 0.4)
    assert np.array_equal(h.view(np.uint32), want.view(np.uint32))
    assert np.array_equal(ch.astype(np.uint64), changes)
