"""The work that programs built on this library have it do, as cases to time.

A case is one call, or one short sequence of calls, through the Python binding
of the C ABI: counting H_k of one graph, loading and counting a graph that has
just arrived, a null-model ensemble with z-scores, making null graphs, serving a
queue of requests, and a program's whole run including the isomorphism table.
Graphs are directed Chung-Lu (power-law) or uniform digraphs of the sizes of the
repository's workloads; their arcs come from the seed alone.

``listed()`` names the cases, ``draw(rng)`` gives others of the same ranges,
``prepare`` makes what a program holds before the call, ``run`` is one pass,
``work`` what a pass cannot do without and ``exact`` the 64-bit reference of the
z-scores (histograms are whole numbers).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1804_09741_gb300 as mt
from paper_1804_09741_gb300.server import Server, run_stream

# Per-direction degree caps of the request stream, by k.
CAPS = {3: 150, 4: 150, 5: 60, 6: 40}


def listed():
    return [
        # the smallest call: a triad census of a 300-vertex network read into a
        # host array, where launches and the host path are all there is
        dict(name="count_k3_small", kind="count", k=3, graph="uniform", n=300, m=1500, gamma=0.0,
             dmax=0, recip=0.0, method=0, compact=False, host=True),
        # a large network that has just been read from disk: load from host CSR,
        # validate, build, count, read out; sizes that are multiples of nothing
        dict(name="load_count_k3_large", kind="load_count", k=3, graph="chung_lu", n=19997,
             m=119983, gamma=2.3, dmax=150, recip=0.15),
        # one count each of the three power-law workload graphs, result left on
        # the GPU: ordinary single-network motif counts
        dict(name="count_k4", kind="count", k=4, graph="chung_lu", n=2000, m=8000, gamma=2.3,
             dmax=150, recip=0.15, method=0, compact=False, host=False),
        dict(name="count_k5", kind="count", k=5, graph="chung_lu", n=1500, m=6000, gamma=2.2,
             dmax=0, recip=0.10, method=0, compact=False, host=False),
        dict(name="count_k6", kind="count", k=6, graph="chung_lu", n=800, m=3200, gamma=2.5,
             dmax=40, recip=0.10, method=0, compact=False, host=False),
        # significance of triads: 511 null graphs of a small network, z-scores
        dict(name="batch_k3_511", kind="batch", k=3, graph="uniform", n=300, m=1500, gamma=0.0,
             dmax=0, recip=0.0, method=0, compact=False, nulls=511, dyads=False),
        # the two null-model workloads, and the k=5 one by the cell method
        dict(name="batch_k5_256", kind="batch", k=5, graph="chung_lu", n=1500, m=6000, gamma=2.2,
             dmax=0, recip=0.10, method=0, compact=False, nulls=256, dyads=False),
        dict(name="batch_k5_256_cells", kind="batch", k=5, graph="chung_lu", n=1500, m=6000,
             gamma=2.2, dmax=0, recip=0.10, method=1, compact=False, nulls=256, dyads=False),
        dict(name="batch_k6_64", kind="batch", k=6, graph="chung_lu", n=800, m=3200, gamma=2.5,
             dmax=40, recip=0.10, method=0, compact=False, nulls=64, dyads=False),
        # one null graph made and read back, for programs that keep their own
        # ensembles
        dict(name="null_graph", kind="null", graph="chung_lu", n=1500, m=6000, gamma=2.2, dmax=0,
             recip=0.10, attempts=60000, dyads=False),
        # a queue of mixed requests through the continuous-batching server
        dict(name="serve_24", kind="serve", requests=24, stream=11, nmax=20000, method=0),
        # a program's whole run on one network: k=6 table, load, count, read out
        # the histogram and the classes it is indexed by
        dict(name="one_shot_k6", kind="one_shot", k=6, graph="chung_lu", n=800, m=3200, gamma=2.5,
             dmax=40, recip=0.10),
    ]


# ------------------------------------------------------------------ graphs


def _weights(n, m, gamma, dmax):
    """Expected degrees of the power law, scaled to sum m and clipped at dmax."""
    w = (np.arange(n) + 1.0) ** (-1.0 / (gamma - 1.0))
    w *= m / w.sum()
    for _ in range(100 if dmax else 0):
        w = np.minimum(w, dmax)
        free = w < dmax
        if abs(w.sum() - m) < 1e-6 * m or not free.any():
            break
        w[free] *= (m - w[~free].sum()) / w[free].sum()
    return w


def _graph(c, seed):
    """Sorted CSR (n, row_ptr, col) with exactly m arcs, no loops, none twice;
    a share `recip` of the arcs in mutual pairs."""
    n, m = c["n"], c["m"]
    rng = np.random.Generator(np.random.PCG64([seed & 0xFFFFFFFF, n, m]))
    if c["graph"] == "uniform":
        key = np.empty(0, np.int64)
        while key.size < m:
            a, b = rng.integers(0, n, 2 * m), rng.integers(0, n, 2 * m)
            key = np.concatenate([key, (a * n + b)[a != b]])
            key = key[np.sort(np.unique(key, return_index=True)[1])]
        key = key[:m]
    else:
        w = _weights(n, m, c["gamma"], c["dmax"])
        w_in = w[rng.permutation(n)]
        c_out, c_in = np.cumsum(w) / w.sum(), np.cumsum(w_in) / w_in.sum()
        mutual = int(round(c["recip"] * m / 2))
        pairs = m - mutual  # unordered pairs: the first `mutual` carry both arcs
        tail = np.empty(0, np.int64)
        head = np.empty(0, np.int64)
        while tail.size < pairs:
            a = np.minimum(np.searchsorted(c_out, rng.random(m + 64)), n - 1)
            b = np.minimum(np.searchsorted(c_in, rng.random(m + 64)), n - 1)
            tail = np.concatenate([tail, a[a != b]])
            head = np.concatenate([head, b[a != b]])
            und = np.minimum(tail, head) * n + np.maximum(tail, head)
            first = np.sort(np.unique(und, return_index=True)[1])
            tail, head = tail[first], head[first]
        tail, head = tail[:pairs], head[:pairs]
        key = np.concatenate([tail * n + head, head[:mutual] * n + tail[:mutual]])
    key = np.sort(key)
    row_ptr = np.zeros(n + 1, np.int32)
    row_ptr[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    return n, row_ptr, (key % n).astype(np.int32)


class _Request:
    """A graph as the server's submit takes it."""

    def __init__(self, n, row_ptr, col):
        self.n, self.row_ptr, self.col = n, row_ptr, col


def _stars(n, m, gamma, dmax, k):
    """Expected number of k-stars, the bulk of a power-law graph's k-sets: what
    keeps drawn cases and requests within bounds."""
    w = _weights(n, m, gamma, dmax)
    d = w + w[np.random.Generator(np.random.PCG64(1)).permutation(n)]
    d = np.minimum(d, n - 1)
    s = np.ones(n)
    for i in range(k - 1):
        s *= np.maximum(d - i, 0.0) / (i + 1)
    return float(s.sum())


def _stream(c):
    """Shapes of a stream of requests: k of weights .2/.3/.3/.2, n log-uniform
    from 100 (to 1,000 at k = 6), mean out-degree 2 to 8."""
    rng = np.random.Generator(np.random.PCG64(c["stream"]))
    out = []
    while len(out) < c["requests"]:
        k = int(rng.choice([3, 4, 5, 6], p=[0.2, 0.3, 0.3, 0.2]))
        top = min(c["nmax"], 1000) if k == 6 else c["nmax"]
        n = int(round(math.exp(rng.uniform(math.log(100), math.log(top)))))
        m = int(round(n * rng.uniform(2.0, 8.0)))
        gamma, recip = float(rng.uniform(2.1, 2.8)), float(rng.uniform(0.0, 0.3))
        if _stars(n, m, gamma, CAPS[k], k) <= (1e8 if k == 6 else 1e9):
            out.append(dict(k=k, graph="chung_lu", n=n, m=m, gamma=gamma, dmax=CAPS[k],
                            recip=recip))
    return out


_tables = {}


def _table(k, compact=False):
    """A program builds a k's table once and counts many graphs with it."""
    if (k, compact) not in _tables:
        _tables[k, compact] = mt.table_build(k, compact=compact)
    return _tables[k, compact]


# ------------------------------------------------------------------ a pass


def _seeds(c, seed):
    return np.random.Generator(np.random.PCG64([seed & 0xFFFFFFFF, 7])).integers(
        1, 1 << 62, c["nulls"], dtype=np.uint64)


def prepare(case, seed):
    c = case
    if c["kind"] == "serve":
        shapes = _stream(c)
        reqs = [(s["k"], _Request(*_graph(s, seed + i))) for i, s in enumerate(shapes)]
        server = Server({k: _table(k) for k in sorted({s["k"] for s in shapes})},
                        method=c["method"])
        return dict(case=c, server=server, requests=reqs)
    n, row_ptr, col = _graph(c, seed)
    if c["kind"] == "one_shot":
        return dict(case=c, csr=(n, row_ptr, col))
    if c["kind"] == "load_count":
        return dict(case=c, csr=(n, row_ptr, col), table=_table(c["k"]))
    g = mt.graph_load_csr(n, row_ptr, col)
    if c["kind"] == "null":
        return dict(case=c, g=g, seed=seed + 1)
    t = _table(c["k"], c["compact"])
    if c["kind"] == "count":
        return dict(case=c, g=g, table=t)
    tuning = mt.make_tuning(method=c["method"]) if c["method"] else None
    # a program makes the handle once and steps it with new seeds again and again;
    # the first step captures the handle's CUDA graph
    batch = mt.Batch(g, t, c["nulls"], 10 * c["m"], tuning, null_model=int(c["dyads"]))
    batch.run(_seeds(c, seed + 1))
    return dict(case=c, g=g, batch=batch, seeds=_seeds(c, seed))


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "count":
        if c["host"]:
            return mt.count_host(state["g"], state["table"])
        if c["method"]:
            return mt.count_tuned(state["g"], state["table"], method=c["method"])
        return mt.count(state["g"], state["table"])
    if kind == "load_count":
        g = mt.graph_load_csr(*state["csr"])
        h = mt.count_host(g, state["table"])
        g.free()
        return h
    if kind == "batch":
        return state["batch"].run(state["seeds"])
    if kind == "null":
        make = mt.randomize_dyads if c["dyads"] else mt.randomize
        r = make(state["g"], state["seed"], c["attempts"])
        csr = r.copy_csr()
        r.free()
        return csr
    if kind == "serve":
        results, _, _ = run_stream(state["server"], state["requests"])
        return [h for _, h, _ in results]
    t = mt.table_build(c["k"])
    g = mt.graph_load_csr(*state["csr"])
    h = mt.count_host(g, t)
    masks = t.class_masks()
    g.free()
    t.free()
    return h, masks


# ------------------------------------------------------------------ work and reference


def work(case):
    """Bytes: the graph's CSR in, histograms, z-scores or null graphs out, the
    table written where a pass builds it.  Operations: of an attempt to swap two
    arcs, two SplitMix64 outputs and four membership tests (about 32)."""
    c = case
    if c["kind"] == "serve":
        parts = [work(dict(s, kind="load_count")) for s in _stream(c)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": 0}
    csr = 4 * (c["n"] + 1 + c["m"])
    if c["kind"] == "null":
        return {"bytes": 2 * csr, "flops": 32 * c["attempts"]}
    hist = 8 * mt.NUM_CLASSES[c["k"]]
    if c["kind"] == "batch":
        return {"bytes": csr + (c["nulls"] + 2) * hist,
                "flops": 32 * 10 * c["m"] * c["nulls"]}
    table = 4 << (c["k"] * (c["k"] - 1)) if c["kind"] == "one_shot" else 0
    return {"bytes": csr + hist + table, "flops": 0}


def _splitmix_index(seeds, i, m):
    """floor(r m / 2^64) of SplitMix64 output i of each seed."""
    z = seeds + np.uint64(((i + 1) * 0x9E3779B97F4A7C15) & (2 ** 64 - 1))
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = z ^ (z >> np.uint64(31))
    lo, hi, m = z & np.uint64(0xFFFFFFFF), z >> np.uint64(32), np.uint64(m)
    return ((hi * m + (lo * m >> np.uint64(32))) >> np.uint64(32)).astype(np.int64)


def _null_adjacency(n, row_ptr, col, seeds, attempts):
    """R+1 adjacency matrices: the graph and its degree-preserving arc-swap nulls,
    every graph's attempts in order."""
    src = np.repeat(np.arange(n), np.diff(row_ptr))
    R, m = seeds.size, col.size
    dst = np.tile(col.astype(np.int64), (R, 1))
    adj = np.zeros((R + 1, n, n), bool)
    adj[:, src, col] = True
    rows = np.arange(R)
    for t in range(attempts):
        e1, e2 = _splitmix_index(seeds, 2 * t, m), _splitmix_index(seeds, 2 * t + 1, m)
        a, b, c, d = src[e1], dst[rows, e1], src[e2], dst[rows, e2]
        ok = ((e1 != e2) & (a != c) & (b != d) & (a != d) & (c != b)
              & ~adj[rows + 1, a, d] & ~adj[rows + 1, c, b])
        r, a, b, c, d, e1, e2 = rows[ok], a[ok], b[ok], c[ok], d[ok], e1[ok], e2[ok]
        adj[r + 1, a, b] = adj[r + 1, c, d] = False
        adj[r + 1, a, d] = adj[r + 1, c, b] = True
        dst[r, e1], dst[r, e2] = d, b
    return adj


def _triad_census(adj):
    """Counts of the 13 weakly connected triads, in ascending order of the least
    6-bit mask over the orderings of the three vertices (row-major adjacency
    without the diagonal)."""
    perms = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]
    place = {(i, j): 2 * i + j - (j > i) for i in range(3) for j in range(3) if i != j}

    def least(code):  # code: 2 bits (forward, backward) of the pairs 01, 12, 02
        arcs = [(x, y) for q, (x, y) in enumerate([(0, 1), (1, 2), (0, 2)]) if code[q] & 1]
        arcs += [(y, x) for q, (x, y) in enumerate([(0, 1), (1, 2), (0, 2)]) if code[q] & 2]
        return min(sum(1 << place[p[x], p[y]] for x, y in arcs) for p in perms)

    codes = [(x, y, z) for x in range(4) for y in range(4) for z in range(4)
             if (x > 0) + (y > 0) + (z > 0) >= 2]
    classes = sorted({least(c) for c in codes})
    hist = np.zeros((adj.shape[0], 13), np.int64)
    for g in range(adj.shape[0]):
        a = torch.from_numpy(adj[g]).to("cuda", torch.float64)
        off = 1.0 - torch.eye(a.shape[0], dtype=torch.float64, device="cuda")
        e = [(1 - a) * (1 - a.T) * off, a * (1 - a.T), a.T * (1 - a), a * a.T]
        # the 54 sums of a graph, each set counted once per ordering of its vertices
        sums = torch.stack([((e[x] @ e[y]) * e[z]).sum() for x, y, z in codes]).round().long()
        for c, s in zip(codes, sums.tolist()):
            hist[g, classes.index(least(c))] += s
    return hist // 6


def exact(case, seed):
    """Histograms and z-scores of a triad ensemble in 64 bits; other cases return
    whole numbers alone, or would take minutes."""
    c = case
    if (c["kind"] != "batch" or c["k"] != 3 or c["dyads"]
            or (c["nulls"] + 1) * c["n"] ** 2 > 5e7 or c["m"] * (c["nulls"] + 200) > 1.1e6):
        return None
    seeds = _seeds(c, seed)
    hist = _triad_census(_null_adjacency(*_graph(c, seed), seeds, 10 * c["m"]))
    null = hist[1:].astype(np.float64)
    mu = null.mean(axis=0)
    sigma = np.sqrt(((null - mu) ** 2).mean(axis=0))
    diff = hist[0] - mu
    with np.errstate(divide="ignore", invalid="ignore"):
        z = np.where(sigma > 0, diff / sigma, np.where(diff == 0, 0.0, np.sign(diff) * np.inf))
    return hist, z


# ------------------------------------------------------------------ drawn cases


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count", "count", "load_count", "batch", "batch", "null", "serve",
                       "one_shot"])
    if kind == "serve":
        return dict(kind=kind, requests=_log(rng, 4, 24), stream=rng.randrange(1 << 30),
                    nmax=_log(rng, 1000, 20000), method=int(rng.random() < 0.25))
    if kind == "null":
        m = _log(rng, 500, 25000)
        return dict(kind=kind, graph="chung_lu", n=max(100, int(m / rng.uniform(2, 8))), m=m,
                    gamma=round(rng.uniform(2.1, 2.8), 2), dmax=150,
                    recip=round(rng.uniform(0, 0.3), 2), attempts=10 * m,
                    dyads=rng.random() < 0.5)
    while True:
        k = rng.choice([3, 4, 5, 6])
        nulls = _log(rng, 4, 511) if kind == "batch" else 0
        top = {3: 60000, 4: 20000, 5: 5000, 6: 1000}[k]
        n = _log(rng, 100, min(top, 5000) if kind == "batch" else top)
        m = int(n * rng.uniform(2.0, 8.0))
        gamma = round(rng.uniform(2.1, 2.8), 2)
        stars = (1 + nulls) * _stars(n, m, gamma, CAPS[k], k)
        if stars <= (1e9 if k == 6 else 2e10) and (1 + nulls) * m <= 1.5e6:
            break
    c = dict(kind=kind, k=k, graph="chung_lu", n=n, m=m, gamma=gamma, dmax=CAPS[k],
             recip=round(rng.uniform(0, 0.3), 2))
    if kind == "count":
        compact = k == 6 and rng.random() < 0.3
        c.update(method=0 if compact else int(rng.random() < 0.3), compact=compact, host=False)
        c["host"] = c["method"] == 0 and rng.random() < 0.5
    elif kind == "batch":
        compact = k == 6 and rng.random() < 0.3
        c.update(method=0 if compact else int(rng.random() < 0.3), compact=compact, nulls=nulls,
                 dyads=rng.random() < 0.3)
    return c
