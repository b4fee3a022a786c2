"""Performance cases: the propagations a user of the library runs.

A case names a graph (uniform sparse "er", skewed "rmat", long-diameter
"grid"), a number of seeds and a call:

  "p"      PROPAGATE-P over a resident graph
  "s"      PROPAGATE-S over a resident graph
  "build"  from a CSR in pinned host memory: graph creation, PROPAGATE-P, free
  "batch"  PROPAGATE-P over a mix of resident graphs, every graph's result

Every output is a whole number (per-round, per-seed counts and the arcs each
round revisits). Sizes are those of bench.py's workloads, of the batched and
serving mixes (n from 1e3 to 2e6, s from 64 to 5,568) and of the tests.
"""
import math

import numpy as np
import torch

import paper_2301_06499_gb300 as pg
from paper_2301_06499_gb300 import inputs


def listed():
    return [
        # the smallest graph of the batched mix, one request: launch latency
        {"name": "er1e3_s64_p", "call": "p", "graph": "er", "n": 1_000, "deg": 8.0, "s": 64},
        # a small social graph
        {"name": "er1e4_s64_p", "call": "p", "graph": "er", "n": 10_000, "deg": 8.0, "s": 64},
        # ragged sizes: seeds that fill neither a word nor a power of two of them
        {"name": "er5e4_s300_s", "call": "s", "graph": "er", "n": 49_999, "deg": 11.0, "s": 300},
        # a directed web graph, the paper's 256 seeds, both variants
        {"name": "rmat22d_s256_p", "call": "p", "graph": "rmat", "scale": 22, "ef": 16.0,
         "directed": True, "s": 256},
        {"name": "rmat22d_s256_s", "call": "s", "graph": "rmat", "scale": 22, "ef": 16.0,
         "directed": True, "s": 256},
        # a social network of two billion arcs: the benchmark workload's size
        {"name": "rmat26u_s512_p", "call": "p", "graph": "rmat", "scale": 26, "ef": 16.0,
         "directed": False, "s": 512},
        # road-like: thousands of sparse rounds
        {"name": "grid1024_s128_p", "call": "p", "graph": "grid", "side": 1024, "s": 128},
        # the serving mix's widest requests (eps = 0.05): 87 words per node
        {"name": "er1e6_s5568_p", "call": "p", "graph": "er", "n": 1_000_000, "deg": 16.0,
         "s": 5568},
        # exact mode: every node a seed
        {"name": "exact_er3e4_p", "call": "p", "graph": "er", "n": 30_000, "deg": 8.0,
         "s": 30_000},
        # graph creation from a host CSR with the propagation it is made for
        {"name": "build_rmat22d_s256", "call": "build", "graph": "rmat", "scale": 22, "ef": 16.0,
         "directed": True, "s": 256},
        # many independent graphs at once
        {"name": "batch_mix30", "call": "batch", "count": 30, "n_hi": 1e5},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("er", "er", "rmat", "rmat", "grid", "wide", "exact", "build", "batch"))
    s = max(1, round(_log(rng, 8, 512)))
    if kind == "er":  # small and ordinary graphs, any number of seeds
        return {"call": rng.choice("ps"), "graph": "er", "n": round(_log(rng, 1e3, 2e6)),
                "deg": round(rng.uniform(4.0, 32.0), 2), "s": s}
    if kind == "rmat":
        return {"call": rng.choice("ps"), "graph": "rmat", "scale": rng.randint(10, 24),
                "ef": round(rng.uniform(8.0, 16.0), 2), "directed": rng.random() < 0.5, "s": s}
    if kind == "grid":
        return {"call": "p", "graph": "grid", "side": round(_log(rng, 40, 900)), "s": s}
    if kind == "wide":
        return {"call": rng.choice("ps"), "graph": "er", "n": round(_log(rng, 1e4, 9e5)),
                "deg": round(rng.uniform(4.0, 16.0), 2), "s": round(_log(rng, 513, 5568))}
    if kind == "exact":
        n = round(_log(rng, 2e3, 2.9e4))
        return {"call": "p", "graph": "er", "n": n, "deg": round(rng.uniform(4.0, 16.0), 2), "s": n}
    if kind == "build":
        return {"call": "build", "graph": "rmat", "scale": rng.randint(10, 21),
                "ef": round(rng.uniform(8.0, 16.0), 2), "directed": rng.random() < 0.5, "s": s}
    return {"call": "batch", "count": rng.randint(4, 30), "n_hi": round(_log(rng, 5e3, 9e4))}


def _graph(case, seed, **kw):
    if case["graph"] == "er":
        return pg.Graph.generate("er", seed, n=case["n"], avg_degree=case["deg"], **kw)
    if case["graph"] == "rmat":
        return pg.Graph.generate("rmat", seed, scale=case["scale"], edge_factor=case["ef"],
                                 directed=case["directed"], **kw)
    return pg.Graph.generate("grid", seed, rows=case["side"], cols=case["side"], p_delete=0.05,
                             **kw)


def _pinned(a):
    t = torch.empty(a.size, dtype=torch.from_numpy(a).dtype, pin_memory=True)
    t.numpy()[:] = a
    return t


def _mix(case):
    """The recipes of a batch: sizes log-spaced from 1e3 nodes to the case's
    largest, kinds and seed counts as the batched mix draws them."""
    for k in range(case["count"]):
        n = round(1e3 * (case["n_hi"] / 1e3) ** ((k + 1) / case["count"]))
        s = inputs.S_CLASSES[(k // 3) % 4]
        yield (("er", "rmat", "grid")[k % 3], n, 4.0 + 28.0 * ((7 * k) % 10) / 10, s)


def prepare(case, seed):
    if case["call"] == "batch":
        b = pg.Batch()
        for k, (kind, n, deg, s) in enumerate(_mix(case)):
            gs = seed * 1_000_003 + k
            if kind == "er":
                g = inputs.er(n, deg, gs)
            elif kind == "rmat":
                g = inputs.rmat(round(math.log2(n)), 8.0 + deg / 4, gs, directed=bool(k & 1))
            else:
                g = inputs.grid(round(n ** 0.5), round(n ** 0.5), 0.05, gs)
            b.add_inputs(g, inputs.seeds(g.n, s, gs + 7))
        return case, b, [_rounds_cap(kind, n ** 0.5) for kind, n, _, _ in _mix(case)]
    if case["call"] == "build":
        g = _graph(case, seed, relabel=False)  # the generator's own order, as on the host
        rp, col = (_pinned(a) for a in g.csr())
        n = g.n
        g.close()
        return case, rp, col, inputs.seeds(n, min(case["s"], n), seed + 1)
    g = _graph(case, seed)
    return case, g, inputs.seeds(g.n, min(case["s"], g.n), seed + 1)


def _rounds_cap(kind, side=0):
    return 48 + (round(4 * side) if kind == "grid" else 0)


def _numbers(res, cap):
    """The result in arrays of a fixed number of rounds (zeros past the last),
    as a program keeps the results of several samples side by side."""
    rows = max(cap, res.rounds + 1)
    counts = np.zeros((rows, res.s), np.int32)
    counts[:res.rounds + 1] = res.counts
    arcs = np.zeros(rows + 1, np.int64)
    arcs[:res.rounds + 2] = res.m_active
    return [counts, arcs]


def run(state):
    case = state[0]
    if case["call"] == "batch":
        _, b, caps = state
        b.run()
        return [x for i, cap in enumerate(caps) for x in _numbers(b.result(i), cap)]
    cap = _rounds_cap(case["graph"], case.get("side", 0))
    if case["call"] == "build":
        _, rp, col, seeds = state
        with pg.Graph.from_csr(rp.numpy(), col.numpy(), directed=case["directed"]) as g:
            return _numbers(pg.propagate_p(g, seeds), cap)
    _, g, seeds = state
    return _numbers((pg.propagate_p if case["call"] == "p" else pg.propagate_s)(g, seeds), cap)


def _sizes(case):
    """Nodes, arcs and rounds of the case's graph, from its recipe."""
    if case["graph"] == "er":
        n, m = case["n"], case["n"] * case["deg"]
        return n, m, 2 + math.log(n) / math.log(case["deg"])
    if case["graph"] == "rmat":
        n = 1 << case["scale"]
        return n, n * case["ef"] * (1 if case["directed"] else 2), 8
    n = case["side"] ** 2
    return n, 3.8 * n, 2 * case["side"]


def work(case):
    """The CSR (64-bit row bounds, 32-bit columns) and the seeds read once, the
    counts written once; one OR per arc and signature word."""
    if case["call"] == "batch":
        w = [work({"call": "p", "graph": kind, "n": n, "deg": deg, "scale": round(math.log2(n)),
                   "ef": 8.0 + deg / 4, "directed": True, "side": round(n ** 0.5), "s": s})
             for kind, n, deg, s in _mix(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    n, m, rounds = _sizes(case)
    s = min(case["s"], n)
    return {"bytes": 8 * n + 4 * m + 4 * s + 4 * s * (rounds + 1), "flops": m * -(-s // 64)}


def _balls(rp, col, seeds):
    """Per-round, per-seed counts and revisited arcs, one sweep a round."""
    n, s = rp.size - 1, seeds.size
    deg = np.diff(rp)
    rows = np.flatnonzero(deg)
    sig = np.zeros((n, s), dtype=bool)
    sig[seeds, np.arange(s)] = True
    new, counts, arcs = sig.copy(), [np.ones(s, np.int64)], [0]
    while True:
        got = np.zeros_like(sig)
        got[rows] = np.logical_or.reduceat(new[col], rp[rows], axis=0)
        arcs.append(int(deg[got.any(axis=1) & ~sig.all(axis=1)].sum()))
        new = got & ~sig
        if not new.any():
            return np.array(counts), np.array(arcs)
        sig |= new
        counts.append(new.sum(axis=0))


def exact(case, seed):
    """Every output is a whole number; the small single graphs are also
    recomputed with sets of Booleans."""
    if case["call"] not in "ps" or case["graph"] == "rmat":
        return None
    n, m, rounds = _sizes(case)
    if m * min(case["s"], n) * rounds > 2e9:
        return None
    _, g, seeds = prepare(case, seed)
    rp, col = g.csr()
    step = seeds.size if case["call"] == "p" else 64
    parts = [_balls(rp, col, seeds[k:k + step]) for k in range(0, seeds.size, step)]
    rows = max([_rounds_cap(case["graph"], case.get("side", 0))] + [len(c) for c, _ in parts])
    counts = np.concatenate([np.pad(c, ((0, rows - len(c)), (0, 0))) for c, _ in parts], axis=1)
    arcs = sum(np.pad(a, (0, rows + 1 - len(a))) for _, a in parts)
    return [counts.astype(np.int32), arcs]
