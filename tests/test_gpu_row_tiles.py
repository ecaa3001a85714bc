"""Row kernels that queue their draws (warp tiles): in-degrees around every bound of the
row classes, counters and gather rounds, widths of one to 32 state words, several sets side
by side, and queues that run full, equal the oracle element by element."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

DEGREES = [0, 1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 255, 256, 257, 511, 700, 1025]
# the persistent loop, a launch per step, and the degree-class kernels (hub rows split, too)
PATHS = [{}, {"persistent": -1}, {"fuse_rows": -1, "hub_min_deg": 512, "hub_chunk": 100}, {"fuse_rows": -1, "vector_words": 4}]


def _degree_graph(n=900, seed=5):
    """Every in-degree of DEGREES on three rows, single-digit ones on the rest."""
    rng = np.random.default_rng(seed)
    d = rng.integers(0, 6, size=n)
    d[:3 * len(DEGREES)] = np.repeat(DEGREES, 3)
    d = d[rng.permutation(n)]
    row_ptr = np.zeros(n + 1, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    return W.Graph(row_ptr, rng.integers(0, n, size=int(row_ptr[-1])).astype(np.int32), "degrees")


def _check(f, g, model, sets, R, T, rng_seed, options, w=None, **prm):
    import torch
    graph = f.Graph(g.row_ptr, g.col_idx)
    if w is not None:
        graph.set_arc_weights(w)
    per_real = options != {}   # (the persistent loop runs without per-realization counts)
    out = f.simulate(graph, model, sets, R, T, rng_seed, per_real=per_real, weighted=w is not None,
                     options=dict(options), **prm)
    torch.cuda.synchronize()
    for i, seeds in enumerate(sets):
        ref = O.simulate(model, g.row_ptr, g.col_idx, seeds, R=R, T=T, rng_seed=rng_seed,
                         **({} if w is None else {"arc_weights": w}), **prm)
        what = (model, R, options, i)
        assert np.array_equal(out["counts"][i].cpu().numpy().astype(np.uint64), ref.counts), what
        assert np.array_equal(out["freq"][i].cpu().numpy().view(np.uint32), ref.freq), what
        if per_real:
            assert np.array_equal(out["per_real"][i].cpu().numpy().view(np.uint32), ref.per_real), what


@pytest.mark.parametrize("path", range(len(PATHS)))
@pytest.mark.parametrize("model", [O.SIR, O.SIS, O.SI, O.SEIR, O.SEIS, O.SWIR, O.IC, O.LT])
def test_every_degree_bound(cuda_lib, model, path):
    g = _degree_graph()
    seeds = W.seed_set(g.n, 60, seed=7)
    for R in (33, 250, 1000):
        _check(cuda_lib, g, model, [seeds], R, 5, 11, PATHS[path], beta=0.04, gamma=0.2, alpha=0.4, mu=0.1, nu=0.5,
               ic_mode=O.IC_CONSTANT, ic_p=0.1)


@pytest.mark.parametrize("path", range(len(PATHS)))
@pytest.mark.parametrize("beta", [0.0, 1e-9, 0.003, 0.3, 1.0])
def test_thresholds_from_never_to_certain(cuda_lib, beta, path):
    """beta = 1e-9 rounds to thresholds of all ones, 0.3 and 1 saturate at small counts."""
    g = _degree_graph(seed=6)
    seeds = W.seed_set(g.n, 300, seed=8)
    for model in (O.SIR, O.SEIS):
        _check(cuda_lib, g, model, [seeds], 96, 4, 12, PATHS[path], beta=beta, gamma=beta, alpha=1.0 - beta)


@pytest.mark.parametrize("path", range(len(PATHS)))
@pytest.mark.parametrize("model,beta", [(O.SIR, 0.01), (O.SIS, 0.6)])
def test_arc_queue_runs_full(cuda_lib, model, beta, path):
    """Half of the nodes infectious in every lane: each arc of the long rows is queued, and
    with beta = 0.6 most lanes are reached by the first arcs of their row."""
    g = _degree_graph(seed=9)
    w = np.random.default_rng(3).uniform(0, 2, size=g.nnz).astype(np.float32)
    w[::7] = 0.0
    _check(cuda_lib, g, model, [W.seed_set(g.n, g.n // 2, seed=10)], 200, 3, 13, PATHS[path], w=w, beta=beta, gamma=0.1)


@pytest.mark.parametrize("path", range(len(PATHS)))
@pytest.mark.parametrize("R,n_sets", [(20, 3), (40, 5), (96, 3)])
def test_sets_side_by_side(cuda_lib, R, n_sets, path):
    """Sets narrower than a thread's or a team's words, and slices that are no power of two."""
    g = _degree_graph(seed=14)
    sets = [W.seed_set(g.n, 40 + i, seed=20 + i) for i in range(n_sets)]
    for model in (O.SIS, O.IC):
        _check(cuda_lib, g, model, sets, R, 4, 15, PATHS[path], beta=0.05, gamma=0.3, ic_mode=O.IC_WEIGHTED_CASCADE)


@pytest.mark.parametrize("R", [64, 600])
def test_graph_between_the_fused_bounds(cuda_lib, R):
    """1.05M to 4.2M state words: one launch per step for both classes, no persistent loop."""
    g = W.ba(70_000, 3, seed=31)
    n_words = g.n * (2 if R == 64 else 32)   # words per set: a power of two
    sets = [W.seed_set(g.n, 50, seed=32 + i) for i in range(12 if R == 64 else 1)]
    assert (1 << 20) < n_words * len(sets) <= (1 << 22)
    _check(cuda_lib, g, O.SIS, sets, R, 3, 16, {}, beta=0.1, gamma=0.1)


@pytest.mark.parametrize("longest", [255, 256])
@pytest.mark.parametrize("R", [500, 1000])
def test_longest_row_of_a_small_graph(cuda_lib, R, longest):
    """The words per thread of a small graph follow from its longest row (below 256 arcs: one,
    and the persistent loop)."""
    rng = np.random.default_rng(31)
    d = rng.integers(0, 6, size=400)
    d[[0, 250]] = longest
    row_ptr = np.zeros(401, dtype=np.int32)
    row_ptr[1:] = np.cumsum(d)
    g = W.Graph(row_ptr, rng.integers(0, 400, size=int(row_ptr[-1])).astype(np.int32), "longest")
    for model in (O.SEIS, O.IC, O.LT, O.SWIR):
        _check(cuda_lib, g, model, [W.seed_set(g.n, 20, seed=32)], R, 5, 16, {}, beta=0.05, gamma=0.2, alpha=0.4, mu=0.1,
               nu=0.5, ic_mode=O.IC_CONSTANT, ic_p=0.1)
