"""The share-out of a small graph's step between warp rows and team rows (csrc/fused_split.h),
compiled for the host: every row has CTAs, the grid fits, and no class is left with a small
part of the CTAs for a large part of the work."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_14895_gb300", "csrc")
PROGRAM = """
#include "fused_split.h"
extern "C" void split(const int32_t *start, int32_t n, int64_t nnz, int ns, int64_t cap, int wr, int tr, int32_t *out) {
    const fsgp::FusedSplit f = fsgp::fused_split(start, n, nnz, ns, cap, wr, tr, 8);
    out[0] = f.warp_rows; out[1] = f.grid_mid; out[2] = f.grid_small;
}
"""


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fused_split")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    lib = ctypes.CDLL(str(d / "t.so"))

    def f(deg, nslices, cap, team_rows):
        bits = np.ceil(np.log2(deg.astype(np.float64) + 1)).astype(int)
        start = np.array([(bits > b).sum() for b in range(33)], dtype=np.int32)   # rows of 2^b in-arcs and more
        out = np.zeros(3, dtype=np.int32)
        lib.split(start.ctypes.data_as(ctypes.c_void_p), len(deg), ctypes.c_int64(int(deg.sum())), nslices, ctypes.c_int64(cap),
                  8, team_rows, out.ctypes.data_as(ctypes.c_void_p))
        return int(out[0]), int(out[1]), int(out[2])
    return f


def _degrees(kind, n):
    rng = np.random.default_rng(7)
    if kind == "er10":
        return rng.poisson(10, n)
    if kind == "er256":
        return rng.poisson(256, n)
    if kind == "dense":
        return np.full(n, 400)
    if kind == "few_long":
        return np.where(np.arange(n) < 6, 60000, rng.integers(0, 9, n))
    return np.minimum((rng.pareto(0.9, n) * 4).astype(np.int64), 60000)   # power law


@pytest.mark.parametrize("cap", [2, 3, 296, 304, 456])
@pytest.mark.parametrize("nslices,team_rows", [(1, 256), (1, 64), (1, 32), (4, 8)])
@pytest.mark.parametrize("kind", ["er10", "er256", "dense", "few_long", "power_law"])
@pytest.mark.parametrize("n", [1, 300, 20_000, 500_000])
def test_no_class_starves(split, kind, n, nslices, team_rows, cap):
    deg = _degrees(kind, n)
    warp_rows, mid, small = split(deg, nslices, cap, team_rows)
    assert 0 <= warp_rows <= n and np.sum(deg >= 256) <= warp_rows
    assert 1 <= mid + small <= cap
    assert (mid > 0) == (warp_rows > 0) and (small > 0) == (warp_rows < n)
    # arcs and 16 per row; a class either has a CTA for all its rows at once, or at least a
    # quarter of the CTAs that its part of the work asks for (degrees are known by bucket only)
    order = np.sort(deg)[::-1]
    work_mid, work_small = [float(x.sum() + 16 * len(x)) for x in (order[:warp_rows], order[warp_rows:])]
    for ctas, rows, per_cta, work in ((mid, warp_rows, 8, work_mid), (small, n - warp_rows, team_rows, work_small)):
        if rows:
            assert ctas >= min(-(-rows * nslices // per_cta), int(0.25 * cap * work / (work_mid + work_small)))
