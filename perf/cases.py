"""Performance cases: what a user of this library has it compute, from the
smallest call to whole decompositions of large graphs.

A case is one operation on one seeded graph:

op        est        kh_estimate (Alg. 1 after the level recursion), every node
          core       kh_core_sampled (Core, Alg. 4) and the removal rounds
          core_exact kh_core_exact (ExactCore) and the removal rounds
          hdeg       kh_hdegree_exact
          counts     kh_sampled_counts, j = 0..10
          request    one request of the server: load the host CSR, set h and the
                     sampling, kh_core_sampled, kh_peel_info, free
family    er         G(n, m): uniform edges
          cl         Chung-Lu power law (social and collaboration graphs)
          rmat       R-MAT, 2^scale nodes, .57/.19/.19/.05 (web-like, hubs)
          grid       a x b lattice with 1% shortcuts (road-like)
          ba         a packed batch of Barabasi-Albert graphs, h mixed in {2, 3, 4}
h, eps    path length; accuracy of the sample budget M (Eq. buffer, delta 0.05)

Graphs are drawn on the GPU from the seed; the handle (context, loaded graph,
h and sampling, output buffers) is what a program keeps between calls.  All
results are whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2112_06154_gb300 import graphgen as gg
from paper_2112_06154_gb300 import khcore as K


def listed():
    return [
        # the smallest call: the estimates of one small graph, where latency counts
        {"name": "est_er2k_h2", "op": "est", "family": "er", "n": 2000, "m": 8000, "h": 2, "eps": 0.5},
        # a small decomposition: hundreds of short rounds, launch-bound
        {"name": "core_er2k_h2", "op": "core", "family": "er", "n": 2000, "m": 8000, "h": 2, "eps": 0.5},
        # a server's request on a road-like graph, host arrays in and out
        {"name": "request_grid_h4", "op": "request", "family": "grid", "a": 143, "b": 151, "h": 4, "eps": 0.5},
        # the social-graph workload at its full size, the paper's main algorithm
        {"name": "core_cl200k_h3", "op": "core", "family": "cl", "n": 200000, "deg": 20.0, "h": 3, "eps": 0.5},
        # the same path at h = 2 and a finer accuracy, ragged size
        {"name": "core_cl50k_h2_eps35", "op": "core", "family": "cl", "n": 49999, "deg": 20.0, "h": 2, "eps": 0.35},
        # a web-like graph with hubs, h = 3
        {"name": "core_rmat18_h3", "op": "core", "family": "rmat", "scale": 18, "h": 3, "eps": 0.5},
        # whole-graph estimates of the largest graph (the bench's size)
        {"name": "est_rmat22_h3", "op": "est", "family": "rmat", "scale": 22, "h": 3, "eps": 0.5},
        # exact 2-degrees of a large graph with hubs
        {"name": "hdeg_rmat20_h2", "op": "hdeg", "family": "rmat", "scale": 20, "h": 2, "eps": 0.5},
        # exact 3-degrees of the social graph
        {"name": "hdeg_cl200k_h3", "op": "hdeg", "family": "cl", "n": 200000, "deg": 20.0, "h": 3, "eps": 0.5},
        # counts at every sampling probability 1 .. 2^-10
        {"name": "counts_cl200k_h2", "op": "counts", "family": "cl", "n": 200000, "deg": 20.0, "h": 2, "eps": 0.5},
        # the exact decomposition the sampled one is compared with
        {"name": "exact_cl50k_h2", "op": "core_exact", "family": "cl", "n": 50001, "deg": 20.0, "h": 2, "eps": 0.5},
        # many small graphs in one call
        {"name": "core_ba96", "op": "core", "family": "ba", "graphs": 96, "n_lo": 100, "n_hi": 8000, "eps": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["est", "core", "core", "core", "request", "hdeg", "counts", "core_exact", "batch"])
    if op == "batch":
        return {"op": "core", "family": "ba", "graphs": _log_int(rng, 8, 96), "n_lo": rng.randint(60, 200),
                "n_hi": _log_int(rng, 1000, 8000), "eps": 0.5}
    h = 2 if op == "core_exact" else rng.choice([2, 3, 4])
    eps = rng.choice([0.5, 0.5, 0.35])
    # core_exact and finer budgets grow fastest with n: smaller sizes for them
    top = 50000 if op == "core_exact" else 50000 if op == "core" and (h == 2 or eps < 0.5) else 200000
    fam = rng.choice(["er", "cl", "cl", "rmat", "grid"])
    case = {"op": op, "family": fam, "h": h, "eps": eps}
    if fam == "er":
        case["n"] = _log_int(rng, 1500, min(top, 60000))
        case["m"] = case["n"] * rng.randint(2, 6)
    elif fam == "cl":
        case["n"] = _log_int(rng, 1500, top if h < 4 or op == "est" else min(top, 60000))
        case["deg"] = round(rng.uniform(5.0, 20.0), 2)
    elif fam == "rmat":
        case["scale"] = rng.randint(11, {"est": 21, "hdeg": 20 if h == 2 else 15, "counts": 19 if h == 2 else 15,
                                         "core_exact": 15}.get(op, 15 if h == 2 else 17))
    else:
        side = math.sqrt(_log_int(rng, 1500, top))
        case["a"] = max(3, int(side * rng.uniform(0.7, 1.4)))
        case["b"] = max(3, int(side * rng.uniform(0.7, 1.0)))
    return case


# ---- graphs, drawn on the GPU -------------------------------------------------

def _csr(n, u, v):
    """Symmetric CSR (rowptr int64, col int32; sorted, no loops, no repeats) of GPU edge lists."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
    lo = torch.div(key, n, rounding_mode="floor")
    both = torch.sort(torch.cat([key, (key - lo * n) * n + lo])).values
    src = torch.div(both, n, rounding_mode="floor")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=u.device)
    rowptr[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rowptr, (both - src * n).to(torch.int32)


def _er(case, g):
    n, m = case["n"], case["m"]
    u = torch.randint(0, n, (m,), generator=g, device="cuda")
    v = torch.randint(0, n, (m,), generator=g, device="cuda")
    return _csr(n, u, v)


def _cl(case, g):
    # weights (i + 10)^(-1/(gamma - 1)), gamma = 2.5, capped at n / 40 (5000 at n = 200k)
    n, deg = case["n"], case["deg"]
    w = (torch.arange(n, dtype=torch.float64, device="cuda") + 10.0) ** (-1.0 / 1.5)
    w = torch.clamp(w * (deg * n / w.sum()), max=max(n / 40.0, 20.0))
    cdf = torch.cumsum(w / w.sum(), 0)
    m = int(round(deg * n / 2.0))
    perm = torch.randperm(n, generator=g, device="cuda")
    ends = [perm[torch.searchsorted(cdf, torch.rand(m, generator=g, dtype=torch.float64, device="cuda"))
                 .clamp_(max=n - 1)] for _ in range(2)]
    return _csr(n, ends[0], ends[1])


def _rmat(case, g):
    scale = case["scale"]
    n, m = 1 << scale, 16 << scale
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        x = torch.rand(m, generator=g, device="cuda")
        u.mul_(2).add_(x >= 0.76)
        v.mul_(2).add_(((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
    perm = torch.randperm(n, generator=g, device="cuda")
    return _csr(n, perm[u], perm[v])


def _grid(case, g):
    a, b = case["a"], case["b"]
    idx = torch.arange(a * b, device="cuda").reshape(a, b)
    u = torch.cat([idx[:, :-1].reshape(-1), idx[:-1].reshape(-1)])
    v = torch.cat([idx[:, 1:].reshape(-1), idx[1:].reshape(-1)])
    k = max(1, round(0.01 * u.numel()))
    s = torch.randint(0, a * b, (2, k), generator=g, device="cuda")
    return _csr(a * b, torch.cat([u, s[0]]), torch.cat([v, s[1]]))


def _ba_batch(case, seed):
    # sizes, attachment and h belong to the case (a server's fixed pool), the edges to the seed
    rng = np.random.default_rng(1004)
    q = case["graphs"]
    ns = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), q)).round().astype(np.int64)
    ms = rng.integers(3, 9, q)
    hs = rng.integers(2, 5, q).astype(np.int32)
    return (*gg.barabasi_albert_batch(ns, ms, seed), hs)


class State:
    """A context, a loaded graph with its settings, and the output buffers."""

    def __init__(self, case, seed):
        K.load()
        self.case = case
        self.ctx = self.graph = None
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        op, h = case["op"], case.get("h", 0)
        if case["family"] == "ba":
            self.ctx = K.kh_ctx_create(0)
            off, rowptr, col, hs = _ba_batch(case, seed)
            self.graph = K.kh_graph_load_batch(self.ctx, off, rowptr, col, hs)
            K.kh_set_sampling(self.graph, seed=seed + 1, M=0, eps=case["eps"])
            n = self.graph.n
        else:
            make = {"er": _er, "cl": _cl, "rmat": _rmat, "grid": _grid}[case["family"]]
            rowptr, col = make(case, g)
            n = rowptr.numel() - 1
            torch.cuda.current_stream().synchronize()
            self.stream = torch.cuda.Stream()
            self.ctx = K.kh_ctx_create(0, self.stream)
            if op == "request":
                self.host = (rowptr.cpu().numpy(), col.cpu().numpy())
                self.seed = seed + 1
                return
            self.graph = K.kh_graph_load_csr(self.ctx, rowptr, col)
            K.kh_set_h(self.graph, h)
            K.kh_set_sampling(self.graph, seed=seed + 1, M=0, eps=case["eps"])
        # small results go to host arrays, large ones stay on the device
        on_host = n < 20000
        types = {"est": [np.uint64, np.uint8, np.int32], "core": [np.uint64], "core_exact": [np.int32],
                 "hdeg": [np.int32], "counts": [np.int32]}[op]
        shape = (n, 11) if op == "counts" else (n,)
        if on_host:
            self.out = [np.zeros(shape, t) for t in types]
        else:
            dev = {np.uint64: torch.int64, np.uint8: torch.uint8, np.int32: torch.int32}
            self.out = [torch.zeros(shape, dtype=dev[t], device="cuda") for t in types]
            torch.cuda.current_stream().synchronize()

    def __del__(self):
        if self.graph is not None:
            self.graph.close()
        if self.ctx is not None:
            self.ctx.close()


def prepare(case, seed):
    return State(case, seed)


def run(state):
    op = state.case["op"]
    if op == "request":
        G = K.kh_graph_load_csr(state.ctx, *state.host)
        try:
            K.kh_set_h(G, state.case["h"])
            K.kh_set_sampling(G, seed=state.seed, M=0, eps=state.case["eps"])
            core = K.kh_core_sampled(G)
            order, rounds, _ = K.kh_peel_info(G, True)
        finally:
            G.close()
        return core, order, rounds
    G = state.graph
    if op == "est":
        return K.kh_estimate(G, *state.out)
    if op == "hdeg":
        return K.kh_hdegree_exact(G, state.out[0])
    if op == "counts":
        return K.kh_sampled_counts(G, 0, 10, state.out[0])
    core = K.kh_core_sampled(G, state.out[0]) if op == "core" else K.kh_core_exact(G, state.out[0])
    order, rounds, _ = K.kh_peel_info(G, True)
    return core, order, rounds


def _size(case):
    """(nodes, adjacency entries) of a case's graph, about."""
    fam = case["family"]
    if fam == "er":
        return case["n"], 2 * case["m"]
    if fam == "cl":
        return case["n"], int(case["deg"] * case["n"])
    if fam == "rmat":
        return 1 << case["scale"], 30 << case["scale"]
    if fam == "grid":
        return case["a"] * case["b"], 4 * case["a"] * case["b"]
    n = case["graphs"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
    return int(n), int(11 * n)


def work(case):
    """The graph read once and the results written once; the arithmetic is integer."""
    n, nnz = _size(case)
    out = {"est": 13, "core": 12, "core_exact": 8, "hdeg": 4, "counts": 44, "request": 12}[case["op"]]
    return {"bytes": 8 * (n + 1) + 4 * nnz + out * n, "flops": 0}


def exact(case, seed):
    """All outputs are whole numbers, compared as they are: no 64-bit values to hold them against."""
    return None
