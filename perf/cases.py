"""Cases that stand for what users of this framework have it do.

The work is community detection on a graph resident in HBM (one call per
graph, or one call for a batch of independent graphs), the same call on host
buffers, the GSP-Leiden variant, the float64 mode, and the phase calls that
programs use on a partition they already hold (its modularity, its
disconnected communities, its super-vertex graph).  Graphs are drawn with
torch from the seed alone, in the shapes of the repository's benchmark
workloads: R-MAT, planted partitions, grids with long-range pairs.
"""
import math

import numpy as np
import torch

from paper_2402_11454_gb300 import gsp

A, B, C_ = 0.57, 0.19, 0.19  # R-MAT quadrants, the fourth takes the rest


def listed():
    return [
        # the smallest call: an interactive query on a small neighbourhood or
        # one customer's graph; latency and launches decide
        {"name": "small", "call": "louvain", "graph": "planted", "n": 611, "k": 13, "degree": 12.0, "p": 0.8},
        # the benchmark's small workload: 10 K vertices, known communities
        {"name": "planted10k", "call": "louvain", "graph": "planted", "n": 10000, "k": 64, "degree": 16.0, "p": 0.8},
        # an ordinary power-law graph (a forum, a citation network) with an
        # odd vertex count
        {"name": "rmat17", "call": "louvain", "graph": "rmat", "n": 100003, "factor": 16},
        # a million-user social network, read from and returned to host memory
        {"name": "host20", "call": "host", "graph": "rmat", "n": 1 << 20, "factor": 16},
        # the benchmark's R-MAT 22 workload
        {"name": "rmat22", "call": "louvain", "graph": "rmat", "n": 1 << 22, "factor": 16},
        # the largest: half a billion stored edges (a web crawl, a large social network)
        {"name": "rmat24", "call": "louvain", "graph": "rmat", "n": 1 << 24, "factor": 16},
        # road-like: high diameter, degree <= 4, segment lengths as weights
        {"name": "grid", "call": "louvain", "graph": "grid", "rows": 2048, "cols": 2048},
        # many independent graphs in one call (one wave repeat, as the
        # benchmark runs its batch)
        {"name": "batch", "call": "batch", "graph": "batch", "graphs": 512},
        # the GSP-Leiden variant: higher modularity for more time
        {"name": "leiden20", "call": "leiden", "graph": "rmat", "n": 1 << 20, "factor": 16},
        # float64 scores on real-valued weights (similarities, distances)
        {"name": "fp64", "call": "fp64", "graph": "planted", "n": 250007, "k": 500, "degree": 20.0, "p": 0.7},
        # judging a partition found elsewhere: its modularity and its
        # internally disconnected communities
        {"name": "evaluate", "call": "evaluate", "graph": "rmat", "n": 1 << 21, "factor": 16},
        # coarsening by a given partition with new real-valued weights
        # (multilevel layouts and solvers, reweighted between their steps):
        # vertex weights, numbering, canonical super-graph
        {"name": "coarsen", "call": "coarsen", "graph": "rmat", "n": 1 << 20, "factor": 16},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["louvain", "louvain", "louvain", "louvain", "host", "batch", "leiden", "fp64", "evaluate",
                       "coarsen"])
    if call == "batch":
        return {"call": call, "graph": "batch", "graphs": _log_uniform(rng, 8, 768)}
    if call == "fp64" or (call == "louvain" and rng.random() < 0.4):
        n = _log_uniform(rng, 500, 1 << 20)
        return {"call": call, "graph": "planted", "n": n, "k": _log_uniform(rng, 4, max(8, n // 40)),
                "degree": rng.uniform(6.0, 32.0), "p": rng.uniform(0.7, 0.9)}
    if call == "louvain" and rng.random() < 0.35:
        return {"call": call, "graph": "grid", "rows": _log_uniform(rng, 24, 3000), "cols": _log_uniform(rng, 24, 3000)}
    hi = {"louvain": 1 << 23, "host": 1 << 21, "leiden": 1 << 21, "evaluate": 1 << 22, "coarsen": 1 << 21}[call]
    return {"call": call, "graph": "rmat", "n": _log_uniform(rng, 1000, hi), "factor": rng.choice([8, 12, 16])}


# ------------------------------------------------------------------- graphs
def _csr(n, u, v, gen, weights):
    """Symmetric CSR of the undirected pairs (u, v): self-loops dropped,
    duplicate pairs merged.  weights: None (unit), (lo, hi) drawn uniformly,
    or an integer k: whole numbers 1..k."""
    keep = u != v
    lo, hi = torch.minimum(u, v)[keep], torch.maximum(u, v)[keep]
    key = torch.sort(lo * n + hi)[0]
    if key.numel():
        first = torch.ones(key.numel(), dtype=torch.bool, device=key.device)
        first[1:] = key[1:] != key[:-1]
        key = key[first]
    lo, hi = key // n, key % n
    both = torch.cat([key, hi * n + lo])
    if weights is None:
        both = torch.sort(both)[0]
        w = torch.ones(both.numel(), dtype=torch.float32, device=key.device)
    else:
        if isinstance(weights, tuple):
            w = torch.rand(key.numel(), generator=gen, device=key.device) * (weights[1] - weights[0]) + weights[0]
        else:
            w = torch.randint(1, weights + 1, (key.numel(),), generator=gen, device=key.device).float()
        both, order = torch.sort(both)
        w = torch.cat([w, w])[order].contiguous()
    src = both // n
    off = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    torch.cumsum(torch.bincount(src, minlength=n), 0, out=off[1:])
    return off, (both % n).to(torch.int32), w


def _rmat(n, factor, gen):
    """factor * n R-MAT samples on the next power of two, those outside the
    n vertices drawn again as uniform pairs."""
    levels = max(1, (n - 1).bit_length())
    E = factor * n
    u = torch.zeros(E, dtype=torch.int64, device="cuda")
    v = torch.zeros(E, dtype=torch.int64, device="cuda")
    for _ in range(levels):
        r = torch.rand(E, generator=gen, device="cuda")
        u.mul_(2).add_(r >= A + B)
        v.mul_(2).add_(((r >= A) & (r < A + B)) | (r >= A + B + C_))
    if n != 1 << levels:
        out = (u >= n) | (v >= n)
        cnt = int(out.sum())
        u[out] = torch.randint(0, n, (cnt,), generator=gen, device="cuda")
        v[out] = torch.randint(0, n, (cnt,), generator=gen, device="cuda")
    return u, v


def _planted(n, k, edges, p, base, gen):
    """Edge samples of planted partitions side by side (per-graph arrays n, k,
    edges, p; base: first vertex): a vertex's community is its index mod k; a
    sample joins two members of one community with probability p, else any
    two vertices of its graph."""
    g = torch.repeat_interleave(torch.arange(n.numel(), device="cuda"), edges)
    E = g.numel()
    r = torch.rand((4, E), generator=gen, device="cuda", dtype=torch.float64)
    ng, kg = n[g], k[g]
    c = torch.minimum((r[1] * kg).long(), kg - 1)
    size = (ng - c + kg - 1) // kg
    intra = r[0] < p[g]
    ends = []
    for q in (r[2], r[3]):
        inside = c + kg * torch.minimum((q * size).long(), size - 1)
        anywhere = torch.minimum((q * ng).long(), ng - 1)
        ends.append(base[g] + torch.where(intra, inside, anywhere))
    return ends[0], ends[1]


def _grid(rows, cols, gen):
    """4-neighbour grid, 5 % of the edges removed, 0.1 % long-range pairs."""
    ids = torch.arange(rows * cols, device="cuda").view(rows, cols)
    u = torch.cat([ids[:, :-1].reshape(-1), ids[:-1, :].reshape(-1)])
    v = torch.cat([ids[:, 1:].reshape(-1), ids[1:, :].reshape(-1)])
    keep = torch.rand(u.numel(), generator=gen, device="cuda") >= 0.05
    extra = torch.randint(0, rows * cols, (2, u.numel() // 1000), generator=gen, device="cuda")
    return torch.cat([u[keep], extra[0]]), torch.cat([v[keep], extra[1]])


def _batch_sizes(graphs):
    """Sizes of the batch's graphs (the same for every seed): vertices
    log-uniform in [64, 65536], 4..64 communities, mean degree 4..64."""
    r = np.random.default_rng(graphs).random((4, graphs))
    n = np.floor(64.0 * 1024.0 ** r[0]).astype(np.int64)
    k = np.minimum(4 + np.floor(61 * r[1]).astype(np.int64), n)
    edges = np.floor(n * (4.0 + 60.0 * r[2]) / 2.0).astype(np.int64)
    return n, k, edges, 0.7 + 0.2 * r[3]


def _sizes(case):
    """Vertices and stored entries (before duplicates merge) of a case."""
    if case["graph"] == "rmat":
        return case["n"], 2 * case["factor"] * case["n"]
    if case["graph"] == "planted":
        return case["n"], 2 * int(case["n"] * case["degree"] / 2)
    if case["graph"] == "grid":
        return case["rows"] * case["cols"], 4 * case["rows"] * case["cols"]
    n, _, edges, _ = _batch_sizes(case["graphs"])
    return int(n.sum()), 2 * int(edges.sum())


def _graph(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["call"] == "coarsen":  # one sparsity pattern and partition, new weights with each seed
        weight_gen, gen = gen, torch.Generator(device="cuda").manual_seed(case["n"])
    else:
        weight_gen = gen
    real = case["call"] in ("fp64", "coarsen")
    weights = (1.0, 10.0) if real else None
    gvo = None
    if case["graph"] == "rmat":
        n = case["n"]
        u, v = _rmat(n, case["factor"], gen)
    elif case["graph"] == "grid":
        n = case["rows"] * case["cols"]
        u, v = _grid(case["rows"], case["cols"], gen)
        weights = 9  # whole lengths
    else:
        if case["graph"] == "planted":
            sizes = (np.array([case["n"]]), np.array([case["k"]]), np.array([int(case["n"] * case["degree"] / 2)]),
                     np.array([case["p"]]))
        else:
            sizes = _batch_sizes(case["graphs"])
        gvo = np.concatenate([[0], np.cumsum(sizes[0])])
        n = int(gvo[-1])
        dev = [torch.from_numpy(x).cuda() for x in sizes + (gvo[:-1],)]
        u, v = _planted(*dev[:4], dev[4], gen)
    return _csr(n, u, v, weight_gen, weights) + (gvo,)


def _follow_partition(off, tgt):
    """A partition as a cheap first guess gives it: every vertex joins its
    neighbour of highest degree (itself when none is higher), twice; heavy-
    tailed sizes, some communities internally disconnected."""
    n = off.numel() - 1
    deg = off[1:] - off[:-1]
    src = torch.repeat_interleave(torch.arange(n, device=off.device), deg)
    key = deg * n + torch.arange(n, device=off.device)
    best = key.clone().scatter_reduce_(0, src, key[tgt.long()], "amax")
    lead = best % n
    return lead[lead].to(torch.int32)


# -------------------------------------------------------------------- cases
def prepare(case, seed):
    off, tgt, w, gvo = _graph(case, seed)
    state = {"call": case["call"], "off": off, "tgt": tgt, "w": w}
    if case["call"] == "host":
        for key in ("off", "tgt", "w"):
            state[key] = state[key].cpu().pin_memory()
        state["membership"] = torch.empty(case["n"], dtype=torch.int32, pin_memory=True)
    elif case["call"] == "batch":
        state["gvo"] = gvo.astype(np.uint64)
    elif case["call"] in ("evaluate", "coarsen"):
        state["C"] = _follow_partition(off, tgt)
    return state


def _found(membership, q, st):
    """The partition, its modularity, and how each pass went (a row per pass,
    10 at most: iterations, vertices, communities)."""
    passes = np.zeros((10, 3), dtype=np.int64)
    passes[:st["passes"]] = np.array([st["iterations"], st["vertices"], st["communities"]]).T
    return {"membership": membership, "modularity": q, "passes": passes}


def run(state):
    call = state["call"]
    graph = (state["off"], state["tgt"], state["w"])
    if call == "louvain":
        return _found(*gsp.louvain(*graph))
    if call == "host":
        return _found(*gsp.louvain_host(*graph, membership=state["membership"]))
    if call == "leiden":
        return _found(*gsp.louvain(*graph, refine=True))
    if call == "fp64":
        return _found(*gsp.louvain(*graph, precision="fp64"))
    if call == "batch":
        return _found(*gsp.louvain_batched(state["gvo"], *graph, wave_repeats=1))
    if call == "evaluate":
        q = gsp.modularity(*graph, state["C"])
        count, flags = gsp.count_disconnected(state["off"], state["tgt"], state["C"])
        return {"modularity": q, "disconnected": count, "flags": flags}
    K, m = gsp.vertex_weights(*graph)
    dense, k = gsp.renumber(state["C"])
    off, tgt, w = gsp.aggregate(*graph, dense, k)
    return {"K": K, "m": m, "dense": dense, "k": k, "off": off, "tgt": tgt, "w": w}


def work(case):
    n, nnz = _sizes(case)
    graph = 8 * (n + 1) + 8 * nnz
    if case["call"] == "evaluate":
        return {"bytes": graph + 4 * n + n, "flops": 2 * nnz}
    if case["call"] == "coarsen":  # the super-graph's size depends on the partition: at least its row ends
        return {"bytes": graph + 4 * n + 12 * n, "flops": 2 * nnz}
    return {"bytes": graph + 4 * n, "flops": 2 * nnz}


def exact(case, seed):
    """The partition a search ends in has no closed form; the values of the
    phase calls have."""
    if case["call"] not in ("evaluate", "coarsen"):
        return None
    off, tgt, w, _ = _graph(case, seed)
    C = _follow_partition(off, tgt).long()
    n = off.numel() - 1
    src = torch.repeat_interleave(torch.arange(n, device=off.device), off[1:] - off[:-1])
    w64 = w.double()
    K = torch.zeros(n, dtype=torch.float64, device=off.device).scatter_add_(0, src, w64)
    total = float(w64.sum())
    cs, ct = C[src], C[tgt.long()]
    if case["call"] == "evaluate":
        sigma = torch.zeros(n, dtype=torch.float64, device=off.device).scatter_add_(0, C, K)
        q = float(w64[cs == ct].sum()) / total - float((sigma * sigma).sum()) / (total * total) if total > 0 else 0.0
        return {"modularity": q, "disconnected": None, "flags": None}
    ids, dense = torch.unique(C, return_inverse=True)
    k = ids.numel()
    key, inv = torch.unique(dense[src] * k + dense[tgt.long()], return_inverse=True)
    sums = torch.zeros(key.numel(), dtype=torch.float64, device=off.device).scatter_add_(0, inv, w64)
    rows = torch.zeros(k + 1, dtype=torch.int64, device=off.device)
    torch.cumsum(torch.bincount(key // k, minlength=k), 0, out=rows[1:])
    return {"K": K, "m": total / 2, "dense": dense.to(torch.int32), "k": k, "off": rows,
            "tgt": (key % k).to(torch.int32), "w": sums}
