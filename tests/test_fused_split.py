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
extern "C" void split(const int32_t *start, int32_t n, int32_t max_deg, int ns, int64_t cap, int wr, int tr, int32_t *out) {
    const fsgp::FusedSplit f = fsgp::fused_split(start, n, max_deg, ns, cap, cap, wr, tr, 8);
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
        lib.split(start.ctypes.data_as(ctypes.c_void_p), len(deg), int(deg.max()), nslices, ctypes.c_int64(cap),
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


@pytest.mark.parametrize("cap", [2, 3, 304, 456])
@pytest.mark.parametrize("nslices,team_rows", [(1, 256), (1, 32), (4, 8)])
@pytest.mark.parametrize("kind", ["er10", "er256", "dense", "few_long", "power_law"])
@pytest.mark.parametrize("n", [1, 20_000, 500_000])
def test_no_class_starves(split, kind, n, nslices, team_rows, cap):
    deg = _degrees(kind, n)
    warp_rows, mid, small = split(deg, nslices, cap, team_rows)
    assert 0 <= warp_rows <= n and np.sum(deg >= 256) <= warp_rows
    assert 1 <= mid + small <= cap
    assert (mid > 0) == (warp_rows > 0) and (small > 0) == (warp_rows < n)
    # rounds of rows, and of eight arcs of each round's longest row: neither class ends later
    # than twice an even end (the best of all shares of the CTAs)
    order = np.sort(deg)[::-1]

    def ends(rows, ctas, per_cta, teams):
        if len(rows) == 0:
            return 0.0
        first = rows[:: max(1, ctas * per_cta // nslices)]
        return 6.0 * len(first) + first.sum() / (8.0 * teams)
    teams = team_rows / 8

    def step(mid, small):
        return max(ends(order[:warp_rows], mid, 8, teams), ends(order[warp_rows:], small, team_rows, 1.0))
    best = step(mid, small)
    if 0 < warp_rows < n:
        best = min(step(m, cap - m) for m in np.unique(np.linspace(1, cap - 1, 40).astype(int)))
    assert step(mid, small) <= 2.0 * best + 40.0


def test_dense_graphs_get_a_warp_per_row(split):
    """Rows of 200 in-arcs: a team's chain would be 25 rounds of eight, a warp's share of it 7."""
    deg = np.random.default_rng(9).poisson(200, 2000)
    assert split(deg, 1, 304, 32) == (2000, 250, 0)
    deg = np.random.default_rng(9).poisson(256, 40_000)   # (many rounds either way)
    assert split(deg, 1, 304, 64)[0] < 40_000


def test_short_rows_do_not_cost_a_round(split):
    """ER, mean degree 12: giving the longer rows a warp each would take a second round."""
    deg = np.random.default_rng(8).poisson(12, 9000)
    warp_rows, mid, small = split(deg, 1, 304, 32)
    assert warp_rows < 50 and mid + small <= 304
    warp_rows, mid, small = split(deg[:3000], 1, 304, 32)   # and where it does not, they get one
    assert warp_rows > 300 and mid + small <= 304
