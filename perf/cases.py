"""Timed cases of the runtime: what a program that uses it has it do, through its public entry points.

Every case keeps a context (or an FMM plan) the way a long-lived program does; one pass queues
new roots on it, runs them and reads the results back.  Sizes come from the repository's bench
workloads, tests and defaults:

* many small recursions at once (a caller that needs the answer, not the throughput);
* batches of fork-join recursions (fib), N-Queens boards with Divergence-Aware Queueing, and the
  unbalanced hashed tree, whose long dependent chains bound it;
* a resident kernel answering a mixed request stream;
* block-mode mergesort from 10^5 ragged keys to 2^26, and the thread-mode Cilksort with 3 queues;
* orientation and clique counting on an R-MAT graph, by orientation and by pivoting;
* the Laplace FMM: the mixed form at the bench size and on a small skewed set, and the FP64 form.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2604_05982_gb300 import gtap as G
from paper_2604_05982_gb300 import runner

MASK64 = (1 << 64) - 1


def listed():
    return [
        # the smallest call: eight recursions of a few dozen to about a thousand tasks each, where
        # launches and host work dominate
        {"name": "fib_small", "kind": "fib", "roots": 8, "n_lo": 8, "n_hi": 14, "queues": 1},
        # a batch of recursions in one launch, about as many tasks as fib(30)
        {"name": "fib_batch", "kind": "fib", "roots": 16, "n_lo": 22, "n_hi": 28, "queues": 1},
        # boards in one launch with four DAQ queues by depth, as the bench's N-Queens workload
        {"name": "queens_daq4", "kind": "queens", "roots": 6, "n_lo": 9, "n_hi": 13, "queues": 4},
        # the bench's hashed tree (2000 root children, near-critical below), a tree per seed
        {"name": "hashed_tree", "kind": "tree", "roots": 1, "children": 2000, "queues": 1},
        # the served mix: requests handed to the resident kernel, answers polled until all are in
        {"name": "served_mix", "kind": "serve", "requests": 400, "fib_hi": 32, "queens_hi": 12, "scale_hi": 14},
        # a ragged sort of a size that one call has in hand, with the default cutoffs
        {"name": "sort_100k", "kind": "sort", "n": 100003, "dist": "uniform", "cutoff": 4096},
        # the bench's sort: 2^26 uniform keys, 65536-key merge pieces
        {"name": "sort_2pow26", "kind": "sort", "n": 1 << 26, "dist": "uniform", "cutoff": 65536},
        # thread-mode Cilksort, three DAQ queues (recursive tasks, serial sorts, serial merges)
        {"name": "cilksort_300k", "kind": "cilksort", "n": 300007, "queues": 3},
        # orientation and the 4-clique count of a graph, four DAQ queues by depth
        {"name": "kclique4_rmat17", "kind": "kclique", "scale": 17, "factor": 16, "k": 4, "algorithm": "orient"},
        # the FMM at the bench size, mixed form
        {"name": "fmm_mixed_uniform_2pow20", "kind": "fmm", "n": 1 << 20, "dist": "uniform", "mixed": True, "order": 6},
        # a small skewed set, mixed form: the tree, list and launch work weigh more
        {"name": "fmm_mixed_plummer_60k", "kind": "fmm", "n": 60001, "dist": "plummer", "mixed": True, "order": 6},
        # the FP64 form
        {"name": "fmm_fp64_plummer_130k", "kind": "fmm", "n": 130003, "dist": "plummer", "mixed": False, "order": 6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fib", "queens", "tree", "serve", "sort", "sort", "cilksort", "kclique", "fmm", "fmm", "fmm"])
    if kind == "fib":
        lo = rng.randint(8, 24)
        return {"kind": kind, "roots": rng.randint(1, 24), "n_lo": lo, "n_hi": min(28, lo + rng.randint(2, 6)),
                "queues": rng.choice([1, 3])}
    if kind == "queens":
        lo = rng.randint(6, 11)
        return {"kind": kind, "roots": rng.randint(2, 8), "n_lo": lo, "n_hi": rng.randint(lo + 1, 13),
                "queues": rng.choice([1, 2, 4])}
    if kind == "tree":
        return {"kind": kind, "roots": rng.randint(1, 6), "children": _log_int(rng, 100, 2000),
                "queues": rng.choice([1, 3])}
    if kind == "serve":
        return {"kind": kind, "requests": _log_int(rng, 40, 400), "fib_hi": rng.randint(22, 32),
                "queens_hi": rng.randint(9, 12), "scale_hi": rng.randint(10, 14)}
    if kind == "sort":
        n = _log_int(rng, 100_000, 1 << 26) | 1
        return {"kind": kind, "n": min(n, (1 << 26) - 1), "dist": rng.choice(["uniform", "few", "runs"]),
                "cutoff": 4096 if n < (1 << 20) else 65536}
    if kind == "cilksort":
        return {"kind": kind, "n": _log_int(rng, 20_000, 300_000) | 1, "queues": rng.choice([1, 3])}
    if kind == "kclique":
        algorithm = rng.choice(["orient", "orient", "pivot"])
        pivot = algorithm == "pivot"
        return {"kind": kind, "scale": rng.randint(10, 13 if pivot else 16), "factor": rng.randint(6, 16),
                "k": rng.randint(4, 6) if pivot else 4, "algorithm": algorithm}
    mixed = rng.random() < 0.67
    return {"kind": "fmm", "n": _log_int(rng, 3_000, 1_000_000 if mixed else 130_000) | 1,
            "dist": rng.choice(["uniform", "plummer"]), "mixed": mixed, "order": rng.choice([4, 6, 6])}


# ---- inputs ----------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & MASK64)
    return g


def _keys(n, dist, seed):
    """uint32 keys as int32 words: uniform; a thousand distinct values; sorted runs of about 1000 keys."""
    g = _gen(seed)
    x = torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device="cuda", dtype=torch.int64)
    if dist == "few":
        x = x % 1000
    elif dist == "runs":
        m = n // 1000 * 1000
        if m:
            x[:m] = x[:m].reshape(-1, 1000).sort(dim=1).values.reshape(-1)
    return x.to(torch.int32)


def _rmat(scale, factor, seed):
    """Undirected simple R-MAT edges (a, b, c = 0.57, 0.19, 0.19), int32 [m, 2] with u < v, sorted."""
    g = _gen(seed)
    m = factor << scale
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for bit in range(scale - 1, -1, -1):
        r = torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
        u += (r >= 0.76).long() << bit
        v += (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).long() << bit
    lo, hi = torch.minimum(u, v), torch.maximum(u, v)
    keep = lo != hi
    key = torch.unique(lo[keep] << scale | hi[keep])
    return torch.stack([key >> scale, key & ((1 << scale) - 1)], dim=1).to(torch.int32).contiguous()


def _points(n, dist, seed):
    """Positions [n, 3] and charges [n] (U(-1, 1)), FP64: the unit cube, or a Plummer sphere cut at r = 10."""
    g = _gen(seed)
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    if dist == "uniform":
        pos = rand(n, 3)
    else:
        r = torch.rsqrt(rand(n + n // 32 + 1024) ** (-2.0 / 3.0) - 1.0)
        r = r[torch.isfinite(r) & (r <= 10.0)][:n]
        ct = 2.0 * rand(n) - 1.0
        st = torch.sqrt(torch.clamp(1.0 - ct * ct, min=0.0))
        ph = 2.0 * math.pi * rand(n)
        pos = torch.stack([r * st * torch.cos(ph), r * st * torch.sin(ph), r * ct], dim=1)
    return pos.contiguous(), 2.0 * rand(n) - 1.0


class Graph:
    """Edges on the GPU and the buffers that their orientation fills."""

    def __init__(self, scale, factor, seed):
        self.n = 1 << scale
        self.edges = _rmat(scale, factor, seed)
        self.m = int(self.edges.shape[0])
        self.off = torch.empty(self.n + 1, dtype=torch.int64, device="cuda")
        # sized for the sampled edges; the first m entries are used (duplicates are dropped)
        self.adj = torch.zeros(factor << scale, dtype=torch.int32, device="cuda")
        self.src = torch.zeros(factor << scale, dtype=torch.int32, device="cuda")
        self.work = torch.empty(4 * self.n + 16, dtype=torch.int32, device="cuda")

    def orient(self):
        G.gtap_kclique_orient(self.edges.data_ptr(), self.m, self.n, self.off.data_ptr(), self.adj.data_ptr(),
                              self.src.data_ptr(), self.work.data_ptr(), 0)

    def args(self, k, threshold, route, algorithm):
        return G.gtap_kclique_args(self.off.data_ptr(), self.adj.data_ptr(), self.src.data_ptr(), 0, self.m, k,
                                   threshold, route, algorithm)


class State:
    """What a program keeps between passes; its context or plan is released when the state is dropped."""

    def __init__(self, case):
        self.case = case
        self.held = None

    def __del__(self):
        if self.held is not None:
            self.held.close()


def prepare(case, seed):
    s = State(case)
    rng = random.Random(int(seed))
    kind = case["kind"]
    if kind == "fib":
        s.held = runner.Context(G.GTAP_MODE_THREAD, case["queues"])
        s.type = s.held.register("fib")
        route = 1 if case["queues"] > 1 else 0
        # the largest once, the rest spread over the range, in an order of the seed
        ns = [case["n_hi"]] + [rng.randint(case["n_lo"], case["n_hi"]) for _ in range(case["roots"] - 1)]
        rng.shuffle(ns)
        s.roots = [G.gtap_fib_args(n, route, 0, 0) for n in ns]
    elif kind == "queens":
        s.held = runner.Context(G.GTAP_MODE_THREAD, case["queues"])
        s.type = s.held.register("nqueens")
        ns = [case["n_hi"]] + [rng.randint(case["n_lo"], case["n_hi"] - 1) for _ in range(case["roots"] - 1)]
        rng.shuffle(ns)
        s.roots = [G.gtap_nqueens_args(n, 1 if case["queues"] > 1 else 0, 0, 0) for n in ns]
    elif kind == "tree":
        s.held = runner.Context(G.GTAP_MODE_THREAD, case["queues"])
        s.type = s.held.register("uts")
        s.roots = [G.gtap_uts_args(rng.getrandbits(32), runner.UTS_THRESHOLD_Q0199, case["children"], 5,
                                   1 if case["queues"] > 1 else 0, 0) for _ in range(case["roots"])]
    elif kind == "serve":
        s.graphs = {}
        for scale in range(10, case["scale_hi"] + 1):
            s.graphs[scale] = Graph(scale, 16, (int(seed) << 5) + scale)
            s.graphs[scale].orient()
        s.held = runner.Context(G.GTAP_MODE_THREAD, 1, pool_bytes=4 << 30, scratch_bytes=1 << 30, max_roots=4096)
        types = {p: s.held.register(p) for p in ("fib", "nqueens", "kclique", "uts")}
        s.requests = []
        for i in range(case["requests"]):
            which = rng.randrange(4)
            if which == 0:
                s.requests.append((types["fib"], G.gtap_fib_args(rng.randint(20, case["fib_hi"]), 0, 0, 0)))
            elif which == 1:
                s.requests.append((types["nqueens"], G.gtap_nqueens_args(rng.randint(8, case["queens_hi"]), 0, 0, 0)))
            elif which == 2:
                scale = rng.randint(10, case["scale_hi"])
                s.requests.append((types["kclique"], s.graphs[scale].args(4, 64, 0, G.GTAP_KCLIQUE_ORIENT)))
            else:
                s.requests.append((types["uts"], G.gtap_uts_args(rng.getrandbits(32), runner.UTS_THRESHOLD_Q0199,
                                                                 rng.randint(100, 2000), 5, 0, 0)))
    elif kind in ("sort", "cilksort"):
        n = case["n"]
        s.src = _keys(n, case.get("dist", "uniform"), seed)
        s.dst = torch.empty_like(s.src)
        s.tmp = torch.empty_like(s.src)
        if kind == "sort":
            s.held = runner.Context(G.GTAP_MODE_BLOCK, 1, pool_bytes=256 << 20, deque_capacity=16384)
            s.type = s.held.register("mergesort")
            s.args = G.gtap_mergesort_args(s.src.data_ptr(), s.dst.data_ptr(), s.tmp.data_ptr(), n, 4096,
                                           case["cutoff"])
        else:
            s.held = runner.Context(G.GTAP_MODE_THREAD, case["queues"])
            s.type = s.held.register("cilksort")
            s.args = G.gtap_cilksort_args(s.src.data_ptr(), s.dst.data_ptr(), s.tmp.data_ptr(), n, 64, 256,
                                          1 if case["queues"] > 1 else 0, 0)
    elif kind == "kclique":
        s.graph = Graph(case["scale"], case["factor"], seed)
        pivot = case["algorithm"] == "pivot"
        s.held = runner.Context(G.GTAP_MODE_THREAD, 4, pool_bytes=1 << 30, scratch_bytes=4 << 30,
                                deque_capacity=16384 if pivot else 4096)
        s.type = s.held.register("kclique")
        s.args = s.graph.args(case["k"], 32 if pivot else 64, 1,
                              G.GTAP_KCLIQUE_PIVOT if pivot else G.GTAP_KCLIQUE_ORIENT)
    else:
        s.pos, s.q = _points(case["n"], case["dist"], seed)
        s.held = runner.Fmm(order=case["order"], leaf_size=64, theta=0.5, mixed=case["mixed"])
    # the inputs are complete before the runtime's own streams read them
    torch.cuda.synchronize()
    return s


# ---- one pass --------------------------------------------------------------------------------


def _answers(c, type_id, roots):
    c.clear()
    handles = [c.spawn(type_id, a) for a in roots]
    c.run()
    return np.array([c.result_u64(h) for h in handles], dtype=np.int64)


def _served(s):
    ctx = s.held.ctx
    answers = np.zeros(len(s.requests), dtype=np.int64)
    index = {}
    G.gtap_serve_start(ctx)
    try:
        sent = done = 0
        while done < len(s.requests):
            while sent < len(s.requests):
                req = G.gtap_submit(ctx, s.requests[sent][0], s.requests[sent][1], 0)
                if req is None:
                    break
                index[req] = sent
                sent += 1
            for req, value, _, _ in G.gtap_poll(ctx):
                answers[index[req]] = value
                done += 1
    finally:
        G.gtap_serve_stop(ctx)
    return answers


def run(state):
    s, kind = state, state.case["kind"]
    if kind in ("fib", "queens"):
        return {"values": _answers(s.held, s.type, s.roots)}
    if kind == "tree":
        v = _answers(s.held, s.type, s.roots)
        return {"nodes": v >> 32, "leaves": v & 0xFFFFFFFF}
    if kind == "serve":
        return {"values": _served(s)}
    if kind in ("sort", "cilksort"):
        s.held.clear()
        s.held.spawn(s.type, s.args)
        s.held.run()
        return {"keys": s.dst}
    if kind == "kclique":
        s.graph.orient()
        return {"count": _answers(s.held, s.type, [s.args]), "off": s.graph.off, "adj": s.graph.adj,
                "src": s.graph.src}
    phi = s.held.run(s.pos, s.q)
    # the mixed form's potentials carry FP32 accuracy: a program that chose it keeps them as FP32
    return {"phi": phi.float() if s.case["mixed"] else phi}


# ---- what a pass cannot do without -----------------------------------------------------------


def _fib(n):
    a, b = 0, 1
    for _ in range(n):
        a, b = b, a + b
    return a


# partial placements of 0..n rows on an n x n board: the tasks of one N-Queens search
_QUEENS_TASKS = {6: 153, 7: 552, 8: 2057, 9: 8394, 10: 35539, 11: 166926, 12: 856189, 13: 4674890}


def work(case):
    """Bytes: inputs once and outputs once.  Flops: one operation per task of a counting program, one
    comparison per key and level of a sort, the near-field and translation arithmetic of an FMM."""
    kind = case["kind"]
    if kind == "fib":
        per = [2 * _fib(n + 1) - 1 for n in range(case["n_lo"], case["n_hi"] + 1)]
        return {"bytes": 24 * case["roots"], "flops": per[-1] + (case["roots"] - 1) * sum(per) / len(per)}
    if kind == "queens":
        per = [_QUEENS_TASKS[n] for n in range(case["n_lo"], case["n_hi"])]
        return {"bytes": 24 * case["roots"],
                "flops": _QUEENS_TASKS[case["n_hi"]] + (case["roots"] - 1) * sum(per) / len(per)}
    if kind == "tree":
        # each root child has 1 / (1 - 5 * 0.199) = 200 nodes below it on average, one hash each
        return {"bytes": 48 * case["roots"], "flops": 10 * 200 * case["children"] * case["roots"]}
    if kind == "serve":
        n = case["requests"] / 4
        fib = [2 * _fib(k + 1) - 1 for k in range(20, case["fib_hi"] + 1)]
        queens = [_QUEENS_TASKS[k] for k in range(8, case["queens_hi"] + 1)]
        edges = [14 << k for k in range(10, case["scale_hi"] + 1)]
        # a 4-clique count tests about 100 candidates for each edge of these graphs
        return {"bytes": 128 * case["requests"] + 12 * sum(edges),
                "flops": n * (sum(fib) / len(fib) + sum(queens) / len(queens) + 100 * sum(edges) / len(edges) +
                              10 * 200 * 1050)}
    if kind in ("sort", "cilksort"):
        return {"bytes": 8 * case["n"], "flops": case["n"] * math.log2(case["n"])}
    if kind == "kclique":
        m = case["factor"] << case["scale"]
        return {"bytes": 8 * m + 8 * m + 8 * (1 << case["scale"]), "flops": 100 * m}
    # p2p: about 5000 near points for each point (9 operations); m2l: about 32 translations for each
    # point, each two operations for every pair of coefficients whose orders add up to at most p
    p, n = case["order"], case["n"]
    pairs = sum((2 * a + 1) * (2 * b + 1) for a in range(p + 1) for b in range(p + 1 - a))
    return {"bytes": (32 + (4 if case["mixed"] else 8)) * n, "flops": n * (9 * min(5000, n) + 64 * pairs)}


def exact(case, seed):
    """The direct sum over all other points in FP64 where it takes a few seconds; counts and sorted
    keys are whole numbers and have no rounding to compare."""
    if case["kind"] != "fmm" or case["n"] > 300_000:
        return None
    pos, q = _points(case["n"], case["dist"], seed)
    phi = torch.empty_like(q)
    n = case["n"]
    step = max(1, (1 << 26) // n)
    for i in range(0, n, step):
        p = pos[i:i + step]
        r2 = torch.zeros(p.shape[0], n, dtype=torch.float64, device=pos.device)
        for d in range(3):
            r2 += (p[:, d:d + 1] - pos[None, :, d]) ** 2
        k = torch.arange(p.shape[0], device=pos.device)
        r2[k, k + i] = math.inf
        phi[i:i + step] = torch.rsqrt(r2) @ q
    return {"phi": phi}
