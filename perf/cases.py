"""Cases for measuring orbit counting through the public calls of the package.

A case is one graph (or one packed batch of graphs) and the call that counts
it. Every graph is made on the GPU from the seed alone, in the families the
library is used on: Erdos-Renyi (the paper's synthetic graphs), R-MAT (skewed,
a few hubs), Chung-Lu (power-law degrees) and dense random graphs.

  call   count     one graph in device memory, non-induced counts
         induced   the same, induced counts
         host      one graph in pinned host memory, counts into pinned memory
         batch     many Chung-Lu graphs packed back to back, one call
  graph  er        n vertices, mean degree d
         rmat      n vertices (ids below n of the next power of two), n * ef
                   edge samples, quadrants (.57, .19, .19, .05)
         chunglu   n vertices, exponent gamma, mean degree d
         dense     n vertices, each pair with probability p
         many      `graphs` Chung-Lu graphs, sizes log-uniform in [lo, hi]
"""
import math

import torch

import paper_2606_29651_gb300 as ni


def listed():
    return [
        # One small graph per call: an interactive query or a loop over many
        # small graphs. Nearly all launches and latency.
        {"name": "er_400", "call": "count", "graph": "er", "n": 400, "d": 20.0},
        # The paper's small synthetic graph, G(2000, 0.01).
        {"name": "er_2000", "call": "count", "graph": "er", "n": 2000, "d": 20.0},
        # A dense graph: long out-lists, many triangles and K4s, every 4-cycle
        # root with hundreds of in-neighbours.
        {"name": "dense_1501", "call": "count", "graph": "dense", "n": 1501, "p": 0.5},
        # A small social-network-like graph.
        {"name": "rmat_14", "call": "count", "graph": "rmat", "n": 1 << 14, "ef": 16},
        # A power-law graph of a few hundred thousand edges, induced counts
        # (the variant most graphlet tools report).
        {"name": "chunglu_100003_induced", "call": "induced", "graph": "chunglu", "n": 100003, "gamma": 2.5, "d": 8.0},
        # One large request of the served mix (millions of edges).
        {"name": "er_350001", "call": "count", "graph": "er", "n": 350001, "d": 12.5},
        # A large, sparse graph with few edges per vertex: the passes over the
        # vertices weigh most, and ids need more than 21 bits.
        {"name": "er_3000001_sparse", "call": "count", "graph": "er", "n": 3000001, "d": 6.0},
        # The benchmark's graph: one million vertices, mean degree 32.
        {"name": "er_1000000", "call": "count", "graph": "er", "n": 1000000, "d": 32.0},
        # The same density from host memory: the graph and the counts cross
        # the host link inside the call.
        {"name": "er_300001_host", "call": "host", "graph": "er", "n": 300001, "d": 32.0},
        # A skewed graph of a few million edges.
        {"name": "rmat_18", "call": "count", "graph": "rmat", "n": 1 << 18, "ef": 16},
        # The benchmark's skewed graph (64 million edges, hubs of 1.6e5).
        {"name": "rmat_22", "call": "count", "graph": "rmat", "n": 1 << 22, "ef": 16},
        # The benchmark's batch: thousands of small graphs in one call.
        {"name": "batch_8192", "call": "batch", "graph": "many", "graphs": 8192, "lo": 50, "hi": 5000,
         "gamma": 2.5, "d": 8.0},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["er", "er", "er_host", "rmat", "rmat", "chunglu", "chunglu", "dense", "many", "many"])
    if kind in ("er", "er_host"):
        n, d = _log_uniform(rng, 300, 1000000), round(rng.uniform(4, 32), 2)
        return {"call": "host" if kind == "er_host" else rng.choice(["count", "count", "induced"]), "graph": "er",
                "n": n, "d": d}
    if kind == "rmat":
        return {"call": rng.choice(["count", "count", "induced"]), "graph": "rmat", "n": _log_uniform(rng, 1 << 10, 1 << 21),
                "ef": rng.randint(8, 16)}
    if kind == "chunglu":
        return {"call": rng.choice(["count", "induced", "host"]), "graph": "chunglu", "n": _log_uniform(rng, 300, 1000000),
                "gamma": round(rng.uniform(2.2, 3.0), 2), "d": round(rng.uniform(4, 32), 2)}
    if kind == "dense":
        return {"call": "count", "graph": "dense", "n": _log_uniform(rng, 100, 2000), "p": round(rng.uniform(0.1, 0.6), 2)}
    lo = _log_uniform(rng, 10, 200)
    return {"call": "batch", "graph": "many", "graphs": _log_uniform(rng, 16, 8192), "lo": lo,
            "hi": lo * rng.randint(4, 25), "gamma": round(rng.uniform(2.2, 3.0), 2), "d": round(rng.uniform(4, 12), 2)}


# ------------------------------------------------------------------- graphs

def _csr(n, u, v):
    """CSR (int32, rows ascending) of the simple undirected graph with edges
    {u, v}: loops and repeats dropped."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    row = torch.div(key, n, rounding_mode="floor")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    rowptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return rowptr.to(torch.int32), (key - row * n).to(torch.int32), row


def _weights(n, gamma, d, device):
    w = torch.arange(1, n + 1, dtype=torch.float64, device=device) ** (-1.0 / (gamma - 1.0))
    w *= n * d / w.sum()
    return _fixed(torch.clamp(w, max=math.sqrt(float(w.sum()))))


def _fixed(w):
    """Weights in units of 2^-20, so that their sums do not depend on the order of addition."""
    return torch.round(w * (1 << 20)).to(torch.int64)


def _below(total, count, gen, device):
    """`count` uniform integers below `total` (a tensor of one value, or one per draw)."""
    x = torch.rand(count, generator=gen, device=device, dtype=torch.float64) * total.to(torch.float64)
    return torch.minimum(x.to(torch.int64), total - 1)


def _edges(case, gen, device):
    n, kind = case["n"], case["graph"]
    if kind == "er":
        k = int(round(n * case["d"] / 2))
        return (torch.randint(0, n, (k,), generator=gen, device=device),
                torch.randint(0, n, (k,), generator=gen, device=device))
    if kind == "dense":
        a = torch.rand((n, n), generator=gen, device=device) < case["p"]
        return torch.nonzero(torch.triu(a, 1), as_tuple=True)
    if kind == "rmat":
        k, scale = n * case["ef"], max(1, math.ceil(math.log2(n)))
        u = torch.zeros(k, dtype=torch.int64, device=device)
        v = torch.zeros(k, dtype=torch.int64, device=device)
        for _ in range(scale):
            r = torch.rand(k, generator=gen, device=device)
            u = 2 * u + (r >= 0.76)
            v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        keep = (u < n) & (v < n)
        return u[keep], v[keep]
    w = _weights(n, case["gamma"], case["d"], device)
    cdf = torch.cumsum(w, 0)
    k = int(cdf[-1]) >> 21
    ends = torch.searchsorted(cdf, _below(cdf[-1], 2 * k, gen, device), right=True)
    return ends[:k], ends[k:]


def _many(case, gen, device):
    """The packed batch: (rowptr, colidx with local ids, vertex and edge offsets).
    The sizes are the case's (evenly spread on a log scale), their order the seed's."""
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    x = (torch.randperm(case["graphs"], generator=gen, device=device) + 0.5) / case["graphs"]
    size = torch.floor(torch.exp(lo + x.to(torch.float64) * (hi - lo))).to(torch.int64)
    vo = torch.zeros(case["graphs"] + 1, dtype=torch.int64, device=device)
    vo[1:] = torch.cumsum(size, 0)
    n = int(vo[-1])
    g = torch.repeat_interleave(torch.arange(case["graphs"], device=device), size)
    w = (torch.arange(n, device=device) - vo[g] + 1).to(torch.float64) ** (-1.0 / (case["gamma"] - 1.0))
    total = torch.zeros(case["graphs"], dtype=torch.int64, device=device).index_add_(0, g, _fixed(w)) / float(1 << 20)
    w = _fixed(torch.minimum(w * (size * case["d"] / total)[g], torch.sqrt(size * case["d"])[g]))
    cdf = torch.cumsum(w, 0)
    end = cdf[vo[1:] - 1]
    begin = torch.cat([torch.zeros(1, dtype=torch.int64, device=device), end[:-1]])
    count = (end - begin) >> 21
    eg = torch.repeat_interleave(torch.arange(case["graphs"], device=device), count)

    def ends():   # an endpoint per edge, drawn by weight within the edge's graph
        return torch.searchsorted(cdf, begin[eg] + _below((end - begin)[eg], len(eg), gen, device), right=True)

    rowptr, colidx, row = _csr(n, ends(), ends())
    eo = rowptr[vo].to(torch.int64)
    return rowptr, (colidx - vo[g[row]]).to(torch.int32), vo, eo


def prepare(case, seed):
    device = torch.device("cuda")
    gen = torch.Generator(device=device).manual_seed(seed)
    if case["call"] == "batch":
        rowptr, colidx, vo, eo = _many(case, gen, device)
        return {"call": "batch", "args": (rowptr, colidx, vo, eo)}
    rowptr, colidx, _ = _csr(case["n"], *_edges(case, gen, device))
    if case["call"] == "host":
        out = torch.empty((case["n"], 15), dtype=torch.int64, pin_memory=True)
        return {"call": "host", "args": (rowptr.cpu().pin_memory(), colidx.cpu().pin_memory(), out)}
    return {"call": case["call"], "args": (rowptr, colidx)}


_CALLS = {"count": ni.count, "induced": ni.count_induced, "host": ni.count_host, "batch": ni.count_batch}


def run(state):
    return _CALLS[state["call"]](*state["args"])


def work(case):
    """The CSR read once and the counts written once (expected sizes)."""
    if case["call"] == "batch":
        lo, hi = case["lo"], case["hi"]
        n = case["graphs"] * (hi - lo) / math.log(hi / lo)
        m = n * case["d"]
    else:
        n = case["n"]
        m = {"er": lambda: n * case["d"], "dense": lambda: n * (n - 1) * case["p"],
             "rmat": lambda: 1.8 * n * case["ef"], "chunglu": lambda: n * case["d"]}[case["graph"]]()
    return {"bytes": 4 * (n + 1) + 4 * m + 120 * n, "flops": 0}


# -------------------------------------------------------------- exact counts

def _dense_counts(a):
    """psi_0 .. psi_14 of every vertex from the adjacency matrix, by counting
    each subgraph's copies at a vertex directly (all values below 2^53)."""
    n = a.shape[0]
    d = a.sum(1)
    c = a @ a
    t = c * a
    tri = t.sum(1) / 2
    off = c - torch.diag(torch.diag(c))
    psi = torch.zeros((n, 15), dtype=torch.float64, device=a.device)
    psi[:, 0] = d
    psi[:, 1] = a @ (d - 1)
    psi[:, 2] = d * (d - 1) / 2
    psi[:, 3] = tri
    psi[:, 4] = a @ (a @ (d - 1)) - d * (d - 1) - 2 * tri
    psi[:, 5] = (d - 1) * (a @ (d - 1)) - 2 * tri
    psi[:, 6] = a @ ((d - 1) * (d - 2) / 2)
    psi[:, 7] = d * (d - 1) * (d - 2) / 6
    psi[:, 8] = (off * (off - 1) / 2).sum(1)
    psi[:, 9] = a @ tri - 2 * tri
    psi[:, 10] = t @ (d - 2)
    psi[:, 11] = tri * (d - 2)
    psi[:, 12] = ((a @ (t - a)) * a).sum(1) / 2
    psi[:, 13] = (t * (t - 1) / 2).sum(1)
    u, v = torch.nonzero(a, as_tuple=True)
    for i in range(0, len(u), 65536):          # K4s through the edge (u, v): edges among the common neighbours
        s = a[u[i:i + 65536]] * a[v[i:i + 65536]]
        psi[:, 14].index_add_(0, u[i:i + 65536], ((s @ a) * s).sum(1) / 6)
    return torch.round(psi).to(torch.int64)


# An induced graphlet with its vertex in orbit j holds _HOLDS[k][j]
# non-induced graphlets on the same vertices with that vertex in orbit k.
_HOLDS = {1: {3: 2}, 2: {3: 1},
          4: {8: 2, 9: 2, 10: 1, 12: 4, 13: 2, 14: 6}, 5: {8: 2, 10: 1, 11: 2, 12: 2, 13: 4, 14: 6},
          6: {9: 1, 10: 1, 12: 2, 13: 1, 14: 3}, 7: {11: 1, 13: 1, 14: 1}, 8: {12: 1, 13: 1, 14: 3},
          9: {12: 2, 14: 3}, 10: {12: 2, 13: 2, 14: 6}, 11: {13: 2, 14: 3}, 12: {14: 3}, 13: {14: 3}}


def _exact_of(rowptr, colidx, induced):
    n = len(rowptr) - 1
    a = torch.zeros((n, n), dtype=torch.float64, device=rowptr.device)
    row = torch.repeat_interleave(torch.arange(n, device=rowptr.device), (rowptr[1:] - rowptr[:-1]).to(torch.int64))
    a[row, colidx.to(torch.int64)] = 1
    psi = _dense_counts(a)
    if induced:
        for k in range(14, -1, -1):
            for j, times in _HOLDS.get(k, {}).items():
                psi[:, k] -= times * psi[:, j]
    return psi


def exact(case, seed):
    if case["call"] == "batch":
        if case["graphs"] > 300 or case["hi"] > 3000:
            return None
        rowptr, colidx, vo, _ = prepare(case, seed)["args"]
        vs, parts = vo.tolist(), []
        for a, b in zip(vs[:-1], vs[1:]):
            p, q = int(rowptr[a]), int(rowptr[b])
            parts.append(_exact_of(rowptr[a:b + 1] - p, colidx[p:q], False))
        return torch.cat(parts)
    n = case["n"]
    m = work(case)["bytes"] / 4 - 31 * n
    if n > 6000 or m * n * n > 4e12:   # the K4 step takes about 2 m n^2 operations in 64 bits
        return None
    rowptr, colidx = (x.cuda() for x in prepare(case, seed)["args"][:2])
    return _exact_of(rowptr, colidx, case["call"] == "induced")
