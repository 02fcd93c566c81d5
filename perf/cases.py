"""Workloads of the Louvain engine, for timing one version of it against another.

A case is a dict of plain values; `prepare` makes its inputs on the GPU from a
seed together with the handle a program keeps, `run` takes one pass through the
public entry points and returns what the path computes.  `kind` says which
entry points a case takes:

  solve        load a graph from device memory (validated, as by default), run,
               read the membership: what a user does with every new graph.
               Synchronous, the default mode, whose results are exact
  sweep        a loaded graph run under several initial tolerances in the
               asynchronous mode (the paper's Section 3.1), Q of each
  batch        many small graphs as one batch: load, run, Q of every graph
  serve        host graphs submitted to the request server, all memberships
  incremental  a changed graph run from the membership it had before
  modularity   exact modularity of a given membership of a loaded graph
  static       the same through the entry point that allocates nothing

Graphs (`graph`): "rmat" (heavy-tailed, ids permuted, isolated vertices, as web
and social graphs), "road" (grid with dropped edges and a few shortcuts, ids in
grid order) and "sbm" (planted partition, ids permuted).  `weights` is the
largest edge weight; large ones need 128-bit gains and 64-bit coarse weights.
"""
import math

import numpy as np
import torch

from paper_2301_12390_gb300 import ASYNC, SYNC, Louvain, Server
from paper_2301_12390_gb300.louvain import modularity_static

DEV = "cuda"
#: The initial tolerances of a sweep.
TOLERANCES = (1.0, 0.1, 0.01, 1e-3, 1e-4, 1e-6, 1e-8, 1e-12)


def listed():
    return [
        # a small graph on its own, where launches and host reads count: the
        # planted partition of 64 blocks of 128
        {"name": "sbm_8k", "kind": "solve", "graph": "sbm", "n": 8192, "degree": 16.6, "weights": 1, "prune": 0},
        # an ordinary social graph (the paper's smallest graphs have about 75,000 vertices and 1M edges)
        {"name": "rmat_75k", "kind": "solve", "graph": "rmat", "n": 75879, "degree": 24.0, "weights": 8, "prune": 0},
        # a mid-size graph with real-valued weights scaled to integers: 128-bit gains; classes in turn
        {"name": "rmat_1m_wide", "kind": "solve", "graph": "rmat", "n": 1 << 20, "degree": 32.0, "weights": 10000,
         "prune": 1, "subrounds": 4},
        # the largest heavy-tailed graph: R-MAT of scale 22, edge factor 16
        {"name": "rmat_4m", "kind": "solve", "graph": "rmat", "n": 1 << 22, "degree": 32.0, "weights": 8, "prune": 1},
        # the largest road grid
        {"name": "road_16m", "kind": "solve", "graph": "road", "n": 4096 * 4096, "degree": 3.6, "weights": 100,
         "prune": 1},
        # colour classes, the option for the best synchronous quality
        {"name": "road_4m_colour", "kind": "solve", "graph": "road", "n": 2048 * 2048, "degree": 3.6, "weights": 100,
         "prune": 1, "colour": 1},
        # the asynchronous mode, pruned, as the benchmark runs it, over the tolerances of the paper's sweep
        {"name": "sweep_rmat_4m", "kind": "sweep", "graph": "rmat", "n": 1 << 22, "degree": 32.0, "weights": 8},
        {"name": "sweep_road_4m", "kind": "sweep", "graph": "road", "n": 2048 * 2048, "degree": 3.6, "weights": 100},
        # many small graphs at once (an eighth of the benchmark's 4,096)
        {"name": "batch_512", "kind": "batch", "graphs": 512, "most": 16384},
        # requests of a thousand to 200,000 vertices, from host memory
        {"name": "serve_48", "kind": "serve", "requests": 48, "most": 200000},
        # a graph that changed by 2% of its edges since its last run
        {"name": "incremental_1m", "kind": "incremental", "graph": "rmat", "n": 1 << 20, "degree": 32.0, "weights": 8},
        # scoring a membership that came from elsewhere
        {"name": "modularity_4m", "kind": "modularity", "graph": "rmat", "n": 1 << 22, "degree": 32.0, "weights": 8},
    ]


def _spread(rng, low, high):
    """A whole number between low and high, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "sweep", "batch", "serve", "incremental", "modularity", "static"])
    if kind == "batch":
        return {"kind": kind, "graphs": _spread(rng, 32, 512), "most": 16384}
    if kind == "serve":
        return {"kind": kind, "requests": rng.choice([4, 9, 15, 23, 31, 48]), "most": 200000}
    graph = rng.choice(["rmat", "road", "sbm"] if kind != "sweep" else ["rmat", "road"])
    low, high = {"solve": (1000, 1 << 22), "sweep": (1 << 19, 1 << 22), "incremental": (10000, 1 << 20),
                 "modularity": (1000, 1 << 22), "static": (1000, 1 << 20)}[kind]
    if graph == "sbm":
        high = min(high, 1 << 20)
    case = {"kind": kind, "graph": graph, "n": _spread(rng, low, high),
            "degree": 3.6 if graph == "road" else round(rng.uniform(8, 32), 1),
            "weights": rng.choice([1, 8, 100, 10000]) if kind != "sweep" else rng.choice([8, 100])}
    if kind == "solve":
        # without pruning every iteration scans the whole graph: for graphs of ordinary size
        case["prune"] = rng.choice([0, 1]) if case["n"] <= 1 << 18 else 1
        case["subrounds"] = rng.choice([0, 0, 4])
        case["colour"] = rng.choice([0, 1]) if graph != "rmat" else 0
        case["stop_rule"] = rng.choice([0, 0, 1])
    return case


# ---------------------------------------------------------------- graphs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62))
    return g


def _randint(g, low, high, m):
    return torch.randint(low, high, (m,), generator=g, device=DEV)


def _csr(n, u, v, wmax, g):
    """Symmetric CSR (offsets int64, columns and weights int32) of the distinct pairs u != v, a weight each."""
    keep = u != v
    u, v = u[keep], v[keep]
    pair = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
    u, v = pair // n, pair % n
    w = _randint(g, 1, wmax + 1, len(pair)).to(torch.int32)
    key, order = torch.sort(torch.cat([pair, v * n + u]))
    col = (key % n).to(torch.int32)
    w = torch.cat([w, w])[order]
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return off, col, w


def _rmat_pairs(n, degree, g):
    """R-MAT endpoints (a, b, c, d = .57, .19, .19, .05) below n, ids permuted."""
    bits = max(1, math.ceil(math.log2(n)))
    m = int(n * degree / 2)
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(bits):
        r = torch.rand(m, generator=g, device=DEV)
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    name = torch.randperm(1 << bits, generator=g, device=DEV)
    return name[u] % n, name[v] % n


def _road_pairs(n, g):
    """A grid of near-square sides, a tenth of its edges dropped, and a shortcut for every thousandth."""
    side = max(2, int(math.isqrt(n)))
    i = torch.arange(n, device=DEV)
    right = i[(i % side != side - 1) & (i + 1 < n)]
    down = i[i + side < n]
    u, v = torch.cat([right, down]), torch.cat([right + 1, down + side])
    keep = torch.rand(len(u), generator=g, device=DEV) >= 0.1
    u, v = u[keep], v[keep]
    extra = max(1, len(u) // 1000)
    return torch.cat([u, _randint(g, 0, n, extra)]), torch.cat([v, _randint(g, 0, n, extra)])


def _blocks_pairs(first, size, p_in, g):
    """Pairs inside the blocks [first, first + size), p_in of each block's pairs."""
    m = torch.round(p_in * size * (size - 1) / 2).long()
    b = torch.repeat_interleave(torch.arange(len(m), device=DEV), m)
    s = size[b].double()
    u = (torch.rand(len(b), generator=g, device=DEV, dtype=torch.float64) * s).long()
    v = (torch.rand(len(b), generator=g, device=DEV, dtype=torch.float64) * s).long()
    return first[b] + u, first[b] + v


def _sbm_pairs(n, degree, g):
    """Blocks of about 128, three quarters of a vertex's edges inside its block, ids permuted."""
    k = max(2, n // 128)
    edge = torch.arange(k + 1, device=DEV) * n // k
    first, size = edge[:-1], (edge[1:] - edge[:-1])
    p_in = torch.full((k,), min(0.5, 0.75 * degree / (n / k)), dtype=torch.float64, device=DEV)
    u, v = _blocks_pairs(first, size, p_in, g)
    m = int(n * degree / 8)
    u, v = torch.cat([u, _randint(g, 0, n, m)]), torch.cat([v, _randint(g, 0, n, m)])
    name = torch.randperm(n, generator=g, device=DEV)
    return name[u], name[v]


def _pairs(case, g):
    n = case["n"]
    if case["graph"] == "rmat":
        return _rmat_pairs(n, case["degree"], g)
    if case["graph"] == "road":
        return _road_pairs(n, g)
    return _sbm_pairs(n, case["degree"], g)


def _log_sizes(count, low, high, g):
    u = torch.rand(count, generator=g, device=DEV, dtype=torch.float64)
    return torch.exp(math.log(low) + u * (math.log(high) - math.log(low))).long()


def _batch(case, seed):
    """Planted partitions of 256 vertices and more, 4 to 64 blocks each, side by side: (graph offsets, CSR)."""
    g = _generator(seed)
    G = case["graphs"]
    n = _log_sizes(G, 256, case["most"], g)
    vo = torch.zeros(G + 1, dtype=torch.int64, device=DEV)
    vo[1:] = torch.cumsum(n, 0)
    k = _randint(g, 4, 65, G)
    p_in = 0.05 + 0.15 * torch.rand(G, generator=g, device=DEV, dtype=torch.float64)
    of = torch.repeat_interleave(torch.arange(G, device=DEV), k)   # graph of every block
    j = torch.arange(len(of), device=DEV) - torch.repeat_interleave(torch.cumsum(k, 0) - k, k)
    first = vo[of] + j * n[of] // k[of]
    size = vo[of] + (j + 1) * n[of] // k[of] - first
    u, v = _blocks_pairs(first, size, p_in[of], g)
    uo, vv = _blocks_pairs(vo[:-1], n, torch.full((G,), 1e-3, dtype=torch.float64, device=DEV), g)
    # ids permuted within each graph
    of_v = torch.repeat_interleave(torch.arange(G, device=DEV), n)
    name = torch.argsort(of_v.double() + torch.rand(len(of_v), generator=g, device=DEV, dtype=torch.float64))
    u, v = name[torch.cat([u, uo])], name[torch.cat([v, vv])]
    return vo, _csr(int(vo[-1]), u, v, 1, g)


def _requests(case, seed):
    """Host graphs, half planted partitions and half R-MAT, average degree 8 to 32, weights 1 to 8."""
    g = _generator(seed)
    count = case["requests"]
    # sizes spread over the logarithm, small and large ones in turn
    sizes = [round(1000 * (case["most"] / 1000) ** ((7 * i % count + 0.5) / count)) for i in range(count)]
    degrees = (8 + 24 * torch.rand(count, generator=g, device=DEV)).tolist()
    out = []
    for i, (n, degree) in enumerate(zip(sizes, degrees)):
        u, v = (_sbm_pairs if i % 2 else _rmat_pairs)(n, degree, g)
        out.append(tuple(a.cpu().numpy() for a in _csr(n, u, v, 8, g)))
    return out


def _given_membership(n, g):
    """Communities of very different sizes."""
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    return (u ** 3 * max(1, n // 16)).to(torch.int32)


def _scored(case, seed):
    g = _generator(seed)
    u, v = _pairs(case, g)
    off, col, w = _csr(case["n"], u, v, case["weights"], g)
    return off, col, w, _given_membership(case["n"], g)


# ------------------------------------------------------------- the cases

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        vo, (off, col, w) = _batch(case, seed)
        return {"kind": kind, "lv": Louvain(mode=ASYNC, prune=1), "graphs": vo, "off": off, "col": col, "w": w}
    if kind == "serve":
        return {"kind": kind, "server": Server(mode=SYNC, prune=1), "requests": _requests(case, seed)}
    if kind in ("modularity", "static"):
        off, col, w, memb = _scored(case, seed)
        state = {"kind": kind, "off": off, "col": col, "w": w, "memb": memb}
        if kind == "modularity":
            torch.cuda.synchronize()
            state["lv"] = Louvain()
            state["lv"].load_csr(off, col, w)
        return state
    g = _generator(seed)
    u, v = _pairs(case, g)
    off, col, w = _csr(case["n"], u, v, case["weights"], g)
    state = {"kind": kind, "off": off, "col": col, "w": w,
             "memb": torch.zeros(case["n"], dtype=torch.int32, device=DEV)}
    if kind == "solve":
        state["lv"] = Louvain(mode=SYNC, prune=case["prune"], subrounds=case.get("subrounds", 0),
                              colour_classes=case.get("colour", 0), stop_rule=case.get("stop_rule", 0))
    elif kind == "sweep":
        torch.cuda.synchronize()
        state["lv"] = Louvain(mode=ASYNC, prune=1)
        state["lv"].load_csr(off, col, w)
    else:   # incremental: the membership found before the last 2% of the edges came
        m = len(u) - len(u) // 50
        old = _csr(case["n"], u[:m], v[:m], case["weights"], g)
        torch.cuda.synchronize()
        state["lv"] = Louvain(mode=SYNC, prune=1)
        state["lv"].load_csr(*old)
        state["lv"].run()
        state["before"] = state["lv"].membership(torch.zeros_like(state["memb"]))
    return state


def _score(q, num, M):
    return {"q": q, "num": [num >> 62, num & ((1 << 62) - 1)], "M": M}


def run(state):
    kind = state["kind"]
    if kind == "static":
        return _score(*modularity_static(state["off"], state["col"], state["w"], state["memb"]))
    if kind == "serve":
        server, requests = state["server"], state["requests"]
        for i, (off, col, w) in enumerate(requests):
            server.submit(i, off, col, w)
        done = {}
        while len(done) < len(requests):
            for r in server.poll(wait_ms=1000):
                done[r["id"]] = r
        return {"memb": np.concatenate([server.membership(i) for i in range(len(requests))]),
                "q": np.array([done[i]["q"] for i in range(len(requests))])}
    lv = state["lv"]
    if kind == "modularity":
        return _score(*lv.modularity_of(state["memb"]))
    if kind == "sweep":
        q = []
        for tolerance in TOLERANCES:
            lv.set_options(tolerance=tolerance)
            lv.run()
            q.append(lv.modularity())
        return np.array(q)
    if kind == "batch":
        lv.load_batch(state["graphs"], state["off"], state["col"], state["w"])
        lv.run()
        q, _, M = lv.batch_modularity()
        return {"q": q, "M": M}
    lv.load_csr(state["off"], state["col"], state["w"])
    if kind == "incremental":
        lv.run_from(state["before"])
    else:
        lv.run()
    num, M = lv.modularity_exact()
    return {"memb": lv.membership(state["memb"]), **_score(lv.modularity(), num, M)}


def exact(case, seed):
    """Modularity in 64 bits; a Louvain run has no value that plain arithmetic gives."""
    if case["kind"] not in ("modularity", "static"):
        return None
    off, col, w, memb = _scored(case, seed)
    memb = memb.long()
    row = torch.repeat_interleave(torch.arange(case["n"], device=DEV), off[1:] - off[:-1])
    w = w.double()
    inside = float(w[memb[row] == memb[col.long()]].sum())
    total = torch.zeros(case["n"], dtype=torch.float64, device=DEV).index_add_(0, memb[row], w)
    M = float(w.sum())
    return {"q": inside / M - float(((total / M) ** 2).sum()), "num": None, "M": None}


def _entries(case):
    """CSR entries of a graph (duplicates of R-MAT pairs left out roughly)."""
    return case["n"] * case["degree"] * (0.95 if case["graph"] == "rmat" else 1.0)


def work(case):
    """Every input array read once, every result written once; a sweep reads its graph for each of its runs.
    One comparison or addition an entry."""
    kind = case["kind"]
    if kind == "batch":
        # vertices log-uniform from 256; a vertex's pairs in its block (n / 22 on the mean) and 1e-3 of the others
        n = case["graphs"] * (case["most"] - 256) / math.log(case["most"] / 256)
        return {"bytes": 8 * n + 8 * n * 57 + 16 * case["graphs"], "flops": n * 57}
    if kind == "serve":
        n = case["requests"] * (case["most"] - 1000) / math.log(case["most"] / 1000)
        return {"bytes": 12 * n + 8 * n * 20, "flops": n * 20}
    entries = _entries(case)
    runs = len(TOLERANCES) if kind == "sweep" else 1
    given = 4 * case["n"] if kind in ("incremental", "modularity", "static") else 0
    result = 4 * case["n"] if kind in ("solve", "incremental") else 24
    return {"bytes": runs * (8 * entries + 8 * case["n"]) + given + result, "flops": runs * entries}
