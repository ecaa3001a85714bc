"""Performance cases: the calls a user of the library makes, over the range of sizes they
are made at.  Inputs are generated on the GPU from a seed; a case is a plain dict.

  listed()            the cases that are always measured
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs and handles a program holds before the call
  run(state)          one call, with its whole results
  work(case)          bytes and floating-point operations the call cannot do without
  exact(case, seed)   float64 results of the calls that return computed floats
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_14895_gb300 import fsgp

MODELS = {"sir": fsgp.SIR, "sis": fsgp.SIS, "ic": fsgp.IC, "lt": fsgp.LT, "si": fsgp.SI,
          "seir": fsgp.SEIR, "seis": fsgp.SEIS, "swir": fsgp.SWIR}
PLANES = {"sir": 2, "sis": 1, "ic": 2, "lt": 2, "si": 1, "seir": 3, "seis": 2, "swir": 3}
COMPARTMENTS = {"seir": 4, "swir": 4}
H, F0 = 64, 8   # width and input features of the surrogate network


# ------------------------------------------------------------------------------- cases

def _sim(name, graph, n, deg, model, R, T, seeds, **kw):
    c = {"call": "simulate", "graph": graph, "n": n, "deg": deg, "model": model, "R": R, "T": T,
         "seeds": seeds, "beta": 0.01, "gamma": 0.05, "weighted": False, "sets": 1,
         "per_real": False, "planes": False}
    if name:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    return [
        # interactive use on a citation-network-sized graph: latency of one small run
        _sim("er10k_sir", "er", 10_000, 10, "sir", 64, 50, 100, beta=0.05, gamma=0.1),
        # the paper's default experiment (1,000 realizations, 100 steps, 10% seeds) on a
        # mid-sized citation network: wide rows of state on a small graph, ragged R
        _sim("ba20k_sir_r1000", "ba", 19_717, 2, "sir", 1000, 100, 1971, gamma=0.005),
        # influence estimation on a social network: independent cascade to quiescence
        _sim("ba1m_ic", "ba", 1_000_000, 5, "ic", 1024, 100, 50),
        # linear thresholds on a social network, odd size, final states kept
        _sim("ba700k_lt", "ba", 700_001, 6, "lt", 500, 100, 50, planes=True),
        # full Monte Carlo epidemics on web-graph-like inputs (the headline workload's shape)
        _sim("rmat24_sir", "rmat", 1 << 24, 16, "sir", 256, 100, 1677),
        # endemic spread that never dies out, node count not a power of two
        _sim("rmat8m_sis", "rmat", 8_000_009, 16, "sis", 256, 100, 800),
        # contact networks with tie strengths
        _sim("rmat4m_weighted", "rmat", 1 << 22, 16, "sir", 256, 100, 419, weighted=True),
        # latent-period epidemic with confidence bands: per-realization curves, ragged R
        _sim("ba250k_seir", "ba", 250_007, 4, "seir", 100, 100, 250, beta=0.05, gamma=0.1, per_real=True),
        # opinion dynamics on a social network
        {"name": "ba1m_hk", "call": "hk", "graph": "ba", "n": 1_000_000, "deg": 5, "R": 64, "T": 30, "eps": 0.25},
        # a service's queue: mixed requests over a pool of graphs
        {"name": "batch_pool", "call": "batch", "graphs": 8, "n_min": 1_000, "n_max": 200_000,
         "requests": 32, "T": 100, "pool": 4},
        # screening candidate seed sets with the learned surrogate
        {"name": "ba500k_screen", "call": "screen", "graph": "ba", "n": 500_000, "deg": 4, "cands": 32, "k": 20},
        # training the surrogate: loss and gradient of one sample
        {"name": "ba300k_grad", "call": "grad", "graph": "ba", "n": 300_007, "deg": 4, "k": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["simulate"] * 7 + ["hk", "batch", "screen", "grad"])
    if kind == "hk":
        return {"call": "hk", "graph": rng.choice(["ba", "er"]), "n": _log_int(rng, 1_000, 1_000_000),
                "deg": rng.randint(3, 6), "R": rng.randint(1, 80), "T": rng.randint(5, 30),
                "eps": round(rng.uniform(0.1, 0.5), 3)}
    if kind == "batch":
        return {"call": "batch", "graphs": rng.randint(2, 8), "n_min": 1_000,
                "n_max": _log_int(rng, 20_000, 200_000), "requests": rng.randint(8, 24), "T": rng.randint(30, 100),
                "pool": rng.randint(0, 1 << 20)}
    if kind == "screen":
        return {"call": "screen", "graph": rng.choice(["ba", "rmat"]), "n": _log_int(rng, 20_000, 600_000),
                "deg": rng.randint(3, 6), "cands": rng.randint(8, 40), "k": rng.randint(5, 40)}
    if kind == "grad":
        return {"call": "grad", "graph": rng.choice(["ba", "rmat"]), "n": _log_int(rng, 20_000, 600_000),
                "deg": rng.randint(3, 6), "k": rng.randint(5, 40)}
    graph = rng.choice(["er", "ba", "rmat"])
    n = _log_int(rng, 1_000, 8_000_000)
    deg = {"er": rng.randint(4, 16), "ba": rng.randint(2, 8), "rmat": rng.randint(8, 16)}[graph]
    model = rng.choice(["sir", "sir", "sis", "sis", "ic", "lt", "si", "seir", "seis", "swir"])
    R, T = _log_int(rng, 32, 1024), _log_int(rng, 20, 100)
    cost = lambda r: T * 32.0 * _words(r) * n * (2 * deg + 16)   # noqa: E731
    while cost(R) > 1.5e12 and R > 32:
        R = max(32, R * 2 // 3)
    while cost(R) > 1.5e12 and n > 1_000:
        n = n * 2 // 3
    return _sim(None, graph, n, deg, model, R, T, max(1, int(n * rng.choice([0.0001, 0.001, 0.01]))),
                beta=round(math.exp(rng.uniform(math.log(0.005), math.log(0.2))), 4),
                gamma=round(rng.uniform(0.02, 0.2), 3),
                weighted=model in ("sir", "sis", "si") and rng.random() < 0.3,
                sets=rng.choice([1, 1, 1, 2, 3]) if R <= 256 else 1,
                per_real=rng.random() < 0.25 and R <= 256, planes=rng.random() < 0.25)


# ----------------------------------------------------------------------- input graphs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _csr(n, src, dst, dedup=False):
    """int32 in-CSR (row = target, sources ascending within a row) of an arc list."""
    key = torch.sort(dst.mul_(n).add_(src)).values
    if dedup:
        key = torch.unique_consecutive(key)
    row = torch.div(key, n, rounding_mode="floor")
    col = (key - row * n).to(torch.int32)
    row_ptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0).to(torch.int32)
    return row_ptr, col


def _er(n, deg, seed):
    """Undirected random graph of mean degree deg, both arc directions."""
    m = n * deg // 2
    e = torch.randint(0, n, (2, m), generator=_gen(seed), device="cuda")
    return _csr(n, torch.cat([e[0], e[1]]), torch.cat([e[1], e[0]]))


def _ba(n, m, seed):
    """Preferential attachment: each new node links to m earlier arc endpoints chosen
    uniformly (each endpoint counts once, so a node in proportion to its degree), both
    arc directions.  Link k picks an earlier endpoint slot r: even slots are the source
    of link r/2, odd ones its target, resolved by following the picks."""
    k = torch.arange((n - 1) * m, device="cuda")
    node = k // m + 1
    span = 2 * m * (node - 1)
    pick = (torch.rand(k.numel(), generator=_gen(seed), device="cuda", dtype=torch.float64) * span).long()
    pick = torch.where(span > 0, torch.minimum(pick, span - 1), torch.full_like(pick, -1))
    slot = pick.clone()
    while True:
        odd = (slot > 0) & (slot % 2 == 1)
        if not bool(odd.any()):
            break
        slot = torch.where(odd, pick[torch.clamp(slot, min=0) // 2], slot)
    target = torch.where(slot < 0, torch.zeros_like(slot), node[torch.clamp(slot, min=0) // 2])
    return _csr(n, torch.cat([node, target]), torch.cat([target, node]), dedup=True)


def _rmat(n, ef, seed, a=0.57, b=0.19, c=0.19):
    """R-MAT arcs (duplicates and self-loops kept) on the next power of two, ids scaled to n."""
    scale = max(1, (n - 1).bit_length())
    e = n * ef
    src = torch.zeros(e, dtype=torch.int64, device="cuda")
    dst = torch.zeros(e, dtype=torch.int64, device="cuda")
    gen = _gen(seed)
    for lo in range(0, e, 1 << 26):
        hi = min(e, lo + (1 << 26))
        s, d = src[lo:hi], dst[lo:hi]
        for _ in range(scale):
            r = torch.rand(hi - lo, generator=gen, device="cuda")
            low = r >= a + b
            s.mul_(2).add_(low)
            d.mul_(2).add_(((r >= a) & ~low) | (r >= a + b + c))
    if n != 1 << scale:
        src = (src * n) >> scale
        dst = (dst * n) >> scale
    return _csr(n, src, dst)


def _arcs(graph, n, deg, seed):
    return {"er": _er, "ba": _ba, "rmat": _rmat}[graph](n, deg, seed)


def _words(R):
    return (R + 31) // 32


def _seed_nodes(rng, n, k):
    return rng.choice(n, size=min(k, n), replace=False).astype(np.int32)


def _theta(seed):
    """He-normal weights of the surrogate's parameter vector, small random biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for f in (F0, H, H):
        parts += [rng.normal(0, math.sqrt(2.0 / (2 * f)), 2 * f * H), rng.normal(0, 0.05, H)]
    parts += [rng.normal(0, math.sqrt(1.0 / H), H), np.zeros(1)]
    return np.concatenate(parts).astype(np.float32)


def _candidates(rng, col, n, cands, k):
    """Seed sets from random to hub-heavy ones (a share of nodes drawn as arc sources)."""
    f = rng.random(cands)
    at = torch.from_numpy(rng.integers(0, col.numel(), size=(cands, k))).cuda()
    hubs = col[at].cpu().numpy()
    return np.where(np.arange(k)[None, :] < np.rint(k * f)[:, None], hubs,
                    rng.integers(0, n, size=(cands, k))).astype(np.int32)


# --------------------------------------------------------------------- prepare and run

def _batch_requests(case, seed):
    """The pool's sizes and request parameters follow from the case; the graphs, seed nodes
    and random keys from the seed."""
    shape, rng = np.random.default_rng(case["pool"]), np.random.default_rng(seed)
    graphs, reqs = [], []
    for i in range(case["graphs"]):
        n = int(round(math.exp(shape.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        kind = "er" if shape.integers(4) == 0 else "ba"
        graphs.append((kind, n, int(shape.integers(4, 17) if kind == "er" else shape.integers(2, 9)), seed * 100 + i))
    for j in range(case["requests"]):
        gi = int(shape.integers(len(graphs)))
        k, model = int(shape.integers(1, 501)), int(shape.integers(4))
        reqs.append({"graph": gi, "model": model, "seeds": _seed_nodes(rng, graphs[gi][1], k),
                     "R": int(shape.choice([32, 64, 128, 256, 512, 1024])), "T": case["T"],
                     "beta": float(shape.uniform(0.005, 0.2)), "gamma": 0.1, "rng_seed": int(rng.integers(1 << 31))})
    return graphs, reqs


def prepare(case, seed):
    call = case["call"]
    st = {"case": case, "seed": seed}
    rng = np.random.default_rng(seed)
    if call == "batch":
        graphs, reqs = _batch_requests(case, seed)
        st["graphs"] = [fsgp.Graph(*_arcs(*g)) for g in graphs]
        st["requests"] = [dict(r, graph=st["graphs"][r["graph"]]) for r in reqs]
        return st
    n = case["n"]
    row_ptr, col = _arcs(case["graph"], n, case["deg"], seed)
    g = st["graph"] = fsgp.Graph(row_ptr, col)
    if call == "simulate":
        if case["weighted"]:
            g.set_arc_weights(torch.rand(col.numel(), generator=_gen(seed + 1), device="cuda") * 2)
        st["sets"] = [_seed_nodes(rng, n, case["seeds"]) for _ in range(case["sets"])]
    elif call == "hk":
        st["h0"] = torch.rand((case["R"], n), generator=_gen(seed + 1), device="cuda") * 2 - 1
    else:
        st["net"] = fsgp.Surrogate()
        st["net"].set_params(_theta(seed))
        st["cand"] = _candidates(rng, col, n, case.get("cands", 1), case["k"])
        if call == "grad":
            st["y"] = torch.rand(n, generator=_gen(seed + 1), device="cuda") ** 3
    return st


def run(st):
    case = st["case"]
    call = case["call"]
    if call == "simulate":
        return fsgp.simulate(st["graph"], MODELS[case["model"]], st["sets"], case["R"], case["T"], st["seed"],
                             beta=case["beta"], gamma=case["gamma"], alpha=0.3, mu=0.05, nu=0.3,
                             weighted=case["weighted"], per_real=case["per_real"], final_planes=case["planes"])
    if call == "hk":
        return fsgp.hk(st["graph"], st["h0"], case["T"], case["eps"])
    if call == "batch":
        out = fsgp.batch_run(st["requests"])
        # two whole results of every request: per-step counts, and per-node frequencies
        return {"counts": torch.cat([o["counts"].reshape(-1) for o in out]),
                "freq": torch.cat([o["freq"].reshape(-1) for o in out]),
                "steps_run": torch.cat([o["steps_run"] for o in out])}
    if call == "screen":
        return st["net"].screen(st["graph"], st["cand"], 0.01, 0.1)
    loss, grad = st["net"].grad(st["graph"], st["cand"][0], 0.05, 0.1, st["y"])
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------- work and float64

def _n_arcs(graph, n, deg):
    return n * deg * (2 if graph == "ba" else 1)


def _sim_bytes(n, e, model, R, T, per_real=False, planes=False, weighted=False):
    """Per step the column indices, row pointers and every state word read and written; a
    cascade tries each arc once in the whole run.  Results written once."""
    p, w, c = PLANES[model], _words(R), COMPARTMENTS.get(model, 3)
    out = 4 * c * n + 8 * (T + 1) * c + (4 * R * (T + 1) * c if per_real else 0) + (4 * p * n * w if planes else 0)
    if model in ("ic", "lt"):
        return 4 * (e + n) + 2 * 4 * p * n * w + out
    return T * ((8 if weighted else 4) * e + 4 * n + 2 * 4 * p * n * w) + out


def work(case):
    call = case["call"]
    if call == "batch":
        graphs, reqs = _batch_requests(case, 1)
        names = ["sir", "sis", "ic", "lt"]
        return {"bytes": sum(_sim_bytes(graphs[r["graph"]][1], _n_arcs(*graphs[r["graph"]][:3]), names[r["model"]],
                                        r["R"], r["T"]) for r in reqs), "flops": 0}
    n, e = case["n"], _n_arcs(case["graph"], case["n"], case["deg"])
    if call == "simulate":
        return {"bytes": case["sets"] * _sim_bytes(n, e, case["model"], case["R"], case["T"], case["per_real"],
                                                   case["planes"], case["weighted"]), "flops": 0}
    if call == "hk":
        return {"bytes": case["T"] * (4 * (e + n) + 8 * n * case["R"]), "flops": 4 * case["T"] * case["R"] * e}
    # forward: columns per layer, activations of each layer written and read (bfloat16)
    fwd = 3 * 4 * (e + n) + n * (2 * F0 + 4 * H + 4 * H + 4)
    flops = 2 * n * H * (2 * F0 + 2 * 2 * H) + e * (F0 + 2 * H)
    if call == "screen":
        return {"bytes": case["cands"] * fwd, "flops": case["cands"] * flops}
    # backward: columns of two adjoint aggregations, activations again, float32 gradients
    # of two layers written and read
    return {"bytes": fwd + 2 * 4 * (e + n) + n * (2 * F0 + 3 * 2 * H + 2 * 8 * H + 4), "flops": 3 * flops}


class _Net:
    """The surrogate network in float64 (torch), on one graph."""

    def __init__(self, row_ptr, col, n, theta):
        self.n, self.col = n, col.long()
        self.deg = (row_ptr[1:] - row_ptr[:-1]).long()
        self.row = torch.repeat_interleave(torch.arange(n, device="cuda"), self.deg)
        self.dout = torch.bincount(self.col, minlength=n)
        self.theta = torch.from_numpy(theta).cuda().double()

    def mean(self, h):
        s = torch.zeros_like(h).index_add(0, self.row, h[self.col])
        return s / self.deg.clamp(min=1).double()[:, None]

    def forward(self, seeds, beta, gamma):
        sd = torch.zeros(self.n, dtype=torch.float64, device="cuda")
        mult = torch.bincount(torch.from_numpy(seeds).cuda().long(), minlength=self.n).double()
        sd[mult > 0] = 1.0
        k = torch.zeros_like(sd).index_add(0, self.row, mult[self.col])
        z = torch.zeros_like(sd)
        h = torch.stack([sd, z + beta, z + gamma, torch.log1p(self.deg.double()), torch.log1p(self.dout.double()),
                         torch.log1p(k), z, z], 1)
        o = 0
        for f in (F0, H, H):
            ws = self.theta[o:o + f * H].view(f, H)
            wn = self.theta[o + f * H:o + 2 * f * H].view(f, H)
            b = self.theta[o + 2 * f * H:o + 2 * f * H + H]
            o += 2 * f * H + H
            h = torch.relu(h @ ws + self.mean(h) @ wn + b)
        return torch.sigmoid(h @ self.theta[o:o + H] + self.theta[o + H])


def _exact_hk(case, seed, row_ptr, col):
    n, eps = case["n"], float(np.float32(case["eps"]))
    h = torch.rand((case["R"], n), generator=_gen(seed + 1), device="cuda") * 2 - 1
    h = h.t().contiguous().double()
    deg = (row_ptr[1:] - row_ptr[:-1]).long()
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    col = col.long()
    for _ in range(case["T"]):
        s, c = torch.zeros_like(h), torch.zeros_like(h)
        for lo in range(0, col.numel(), 1 << 22):
            i, j = row[lo:lo + (1 << 22)], col[lo:lo + (1 << 22)]
            hj = h[j]
            near = ((h[i] - hj).abs() < eps).double()
            s.index_add_(0, i, hj * near)
            c.index_add_(0, i, near)
        h = torch.where(c > 0, s / c.clamp(min=1), h)
    return (h.t().contiguous(), None)   # laid out as hk() returns: opinions, change counts


def exact(case, seed):
    call = case["call"]
    if call in ("simulate", "batch"):
        return None   # whole numbers only
    n = case["n"]
    row_ptr, col = _arcs(case["graph"], n, case["deg"], seed)
    if call == "hk":
        return _exact_hk(case, seed, row_ptr, col)
    cand = _candidates(np.random.default_rng(seed), col, n, case.get("cands", 1), case["k"])
    net = _Net(row_ptr, col, n, _theta(seed))
    if call == "screen":
        with torch.no_grad():
            return torch.stack([net.forward(c, 0.01, 0.1).sum() for c in cand])
    net.theta.requires_grad_(True)
    y = (torch.rand(n, generator=_gen(seed + 1), device="cuda") ** 3).double()
    loss = ((net.forward(cand[0], 0.05, 0.1) - y) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach(), "grad": net.theta.grad}
