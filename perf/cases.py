"""The work a user has this engine do, as cases that can be timed.

Every case goes through the package's public `Context`: load graphs, then
count, enumerate, batch or serve.  Inputs are synthetic graphs of the shapes
the repository's own workloads have (sparse and dense random graphs,
power-law interaction networks, molecules), drawn here from the case and a
seed.  Search sizes are heavy-tailed, so as in the paper's experiments, which
set aside instances over a time limit, a pattern whose search lies outside the
case's range of states is set aside while the inputs are prepared.
"""
from __future__ import annotations

import math

import numpy as np

import paper_1705_09358_gb300 as sge

RI, RIDS, SI, SIFC = sge.SGE_RI, sge.SGE_RIDS, sge.SGE_RIDS_SI, sge.SGE_RIDS_SI_FC


def listed():
    return [
        # one interactive query on a sparse graph of a thousand vertices: latency
        {"name": "one_query", "kind": "query", "algo": RI, "n": 1000, "degree": 8, "labels": 8, "k": 8},
        # the matches themselves, listed: a labelled motif with some ten thousand embeddings
        {"name": "list_matches", "kind": "list", "algo": RI, "n": 2003, "degree": 8, "labels": 4, "k": 6},
        # five heavy patterns on a dense target that stays loaded, the strongest pruning: throughput
        {"name": "dense_batch", "kind": "dense", "algo": SIFC, "n": 2000, "degree": 100, "labels": 4, "pats": 5,
         "k_lo": 16, "k_hi": 24, "load": False},
        # the same kind of job from host arrays to results: load, count, unload
        {"name": "dense_load_count", "kind": "dense", "algo": SIFC, "n": 1777, "degree": 89, "labels": 4, "pats": 3,
         "k_lo": 16, "k_hi": 22, "load": True},
        # a dense target of several bitset words per lane, plain RI
        {"name": "dense_wide", "kind": "dense", "algo": RI, "n": 5003, "degree": 120, "labels": 6, "pats": 4,
         "k_lo": 10, "k_hi": 16, "load": False},
        # deep patterns (32 to 64 vertices) on an interaction network of ten thousand proteins
        {"name": "deep", "kind": "network", "algo": SIFC, "n": 10007, "degree": 20, "labels": 32, "pats": 10,
         "k_lo": 32, "k_hi": 64, "serve": False},
        # substructure screening: every pattern against every molecule of a library, edge-labelled
        {"name": "molecules_ri", "kind": "molecules", "algo": RI, "targets": 200, "pats": 1000},
        {"name": "molecules_sifc", "kind": "molecules", "algo": SIFC, "targets": 121, "pats": 601},
        # a batch of queries of 8 to 128 vertices on one large interaction network
        {"name": "network_ri", "kind": "network", "algo": RI, "n": 100000, "degree": 16, "labels": 64, "pats": 160,
         "k_lo": 8, "k_hi": 128, "serve": False},
        {"name": "network_sifc", "kind": "network", "algo": SIFC, "n": 70001, "degree": 16, "labels": 64, "pats": 64,
         "k_lo": 8, "k_hi": 96, "serve": False},
        # the same kind of queries submitted one by one to the serving loop and drained
        {"name": "network_serve", "kind": "network", "algo": RI, "n": 50021, "degree": 16, "labels": 64, "pats": 96,
         "k_lo": 8, "k_hi": 64, "serve": True},
        # directed, edge-labelled motifs (regulation networks)
        {"name": "directed", "kind": "directed", "algo": RIDS, "n": 3001, "degree": 12, "labels": 2, "elabels": 3,
         "pats": 24, "k_lo": 5, "k_hi": 9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "list", "dense", "network", "molecules", "directed"])
    algo = rng.choice([RI, RIDS, SI, SIFC])
    if kind == "query":
        return {"kind": kind, "algo": algo, "n": _log_int(rng, 60, 30000), "degree": rng.randint(4, 10),
                "labels": rng.randint(6, 24), "k": rng.randint(3, 12)}
    if kind == "list":
        return {"kind": kind, "algo": algo, "n": _log_int(rng, 500, 6000), "degree": rng.randint(6, 9),
                "labels": rng.randint(3, 5), "k": rng.randint(4, 7)}
    if kind == "dense":
        k_lo = rng.randint(10, 18)
        return {"kind": kind, "algo": algo, "n": _log_int(rng, 400, 8000), "degree": rng.randint(60, 120),
                "labels": rng.randint(4, 6), "pats": rng.randint(1, 6), "k_lo": k_lo, "k_hi": k_lo + rng.randint(0, 8),
                "load": rng.random() < 0.3}
    if kind == "network":
        k_lo = rng.randint(8, 32)
        return {"kind": kind, "algo": algo, "n": _log_int(rng, 8000, 100000), "degree": rng.randint(14, 20),
                "labels": rng.randint(32, 64), "pats": _log_int(rng, 6, 96), "k_lo": k_lo,
                "k_hi": _log_int(rng, k_lo, 128), "serve": rng.random() < 0.3}
    if kind == "molecules":
        return {"kind": kind, "algo": algo, "targets": _log_int(rng, 8, 160), "pats": _log_int(rng, 20, 800)}
    return {"kind": kind, "algo": algo, "n": _log_int(rng, 300, 6000), "degree": rng.randint(8, 12), "labels": 2,
            "elabels": rng.randint(3, 4), "pats": _log_int(rng, 3, 32), "k_lo": rng.randint(4, 6),
            "k_hi": rng.randint(6, 9)}


# ------------------------------------------------------------------- graphs
class Graph:
    """An edge list with labels, as `Context.load_target` and `load_pattern` take it."""

    def __init__(self, n, src, dst, vlabel, elabel=None, directed=False):
        self.n, self.directed = int(n), directed
        self.src, self.dst, self.vlabel = (np.ascontiguousarray(a, dtype=np.int32) for a in (src, dst, vlabel))
        self.elabel = None if elabel is None else np.ascontiguousarray(elabel, dtype=np.int32)


class Rows:
    """Neighbour rows of a graph (edges both ways), with each entry's edge index."""

    def __init__(self, g):
        u, v = np.concatenate([g.src, g.dst]), np.concatenate([g.dst, g.src])
        order = np.argsort(u.astype(np.int64) * g.n + v, kind="stable")
        self.ptr = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=g.n))])
        self.nbr = v[order]
        self.edge = order % max(1, g.src.shape[0])

    def row(self, v):
        return self.nbr[self.ptr[v]:self.ptr[v + 1]]


def _pairs(r, n, m, ends, directed=False):
    """m distinct loop-free vertex pairs, both endpoints drawn by `ends(count)`."""
    keys = np.zeros(0, np.int64)
    while keys.shape[0] < m:
        want = int((m - keys.shape[0]) * 1.2) + 64
        a, b = ends(want).astype(np.int64), ends(want).astype(np.int64)
        lo, hi = (a, b) if directed else (np.minimum(a, b), np.maximum(a, b))
        keys = np.unique(np.concatenate([keys, (lo * n + hi)[a != b]]))
    keys = r.permutation(keys)[:m]
    return keys // n, keys % n


def _random_graph(r, n, degree, labels, directed=False, elabels=0):
    """Uniform random graph of mean degree `degree` (out-degree if directed), uniform labels."""
    m = min(n * degree // (1 if directed else 2), n * (n - 1) // 4)
    s, d = _pairs(r, n, m, lambda c: r.integers(0, n, c), directed)
    return Graph(n, s, d, r.integers(0, labels, n), r.integers(1, elabels + 1, m) if elabels else None, directed)


def _network(r, n, degree, labels):
    """Power-law graph (exponent 2.2, hubs capped at sqrt(n * degree)) with Zipf(1.1) labels."""
    w = np.arange(1, n + 1, dtype=np.float64) ** (-1.0 / 1.2)
    for _ in range(20):
        w = np.minimum(w * (degree * n / w.sum()), math.sqrt(n * degree))
    cum = np.cumsum(w)
    s, d = _pairs(r, n, n * degree // 2, lambda c: np.minimum(np.searchsorted(cum, r.random(c) * cum[-1]), n - 1))
    p = np.arange(1, labels + 1, dtype=np.float64) ** -1.1
    return Graph(n, s, d, r.choice(labels, n, p=p / p.sum()))


def _molecule(r):
    """Near-tree of 20 to 500 atoms, degree at most 4, a tenth as many ring closures (five- and six-rings)."""
    n = int(r.integers(20, 501))
    deg, parent, edges = [0] * n, [-1] * n, {}
    coin = r.random(4 * n)
    for i in range(1, n):
        j = int(coin[i] * i)
        while deg[j] >= 4:
            j = j + 1 if j + 1 < i else 0
        parent[i] = j
        edges[(j, i)] = 1
        deg[i] += 1
        deg[j] += 1
    for c in range(n // 10):
        a = b = int(coin[n + 2 * c] * n)
        for _ in range(4 if coin[n + 2 * c + 1] < 0.5 else 5):
            b = parent[b] if b > 0 else b
        if deg[a] < 4 and deg[b] < 4 and a != b and (b, a) not in edges:
            edges[(b, a)] = 1
            deg[a] += 1
            deg[b] += 1
    s, d = np.array(list(edges), dtype=np.int32).T
    tail = 0.5 ** np.arange(9)
    p = np.concatenate([[0.60, 0.15, 0.15], 0.10 * tail / tail.sum()])
    return Graph(n, s, d, r.choice(12, n, p=p / p.sum()), r.choice([1, 2, 3], s.shape[0], p=[0.80, 0.15, 0.05]))


# ----------------------------------------------------------------- patterns
def _induced(g, rows, verts):
    pos = {v: i for i, v in enumerate(verts)}
    seen = {}
    for v in verts:
        for t in range(rows.ptr[v], rows.ptr[v + 1]):
            if int(rows.nbr[t]) in pos:
                seen[int(rows.edge[t])] = 1
    e = np.array(sorted(seen), dtype=np.int64)
    src = [pos[int(v)] for v in g.src[e]]
    dst = [pos[int(v)] for v in g.dst[e]]
    return Graph(len(verts), src, dst, g.vlabel[verts], None if g.elabel is None else g.elabel[e], g.directed)


def _walk_pattern(r, g, rows, k):
    """The subgraph on the first k vertices a random walk meets (fewer where it is shut in)."""
    cur = int(r.integers(0, g.n))
    seen = {cur: 1}
    for x in r.random(40 * k):
        if len(seen) == k:
            break
        row = rows.row(cur)
        if row.shape[0] == 0:
            cur = int(x * g.n)
            seen = {cur: 1}
            continue
        cur = int(row[int(x * row.shape[0])])
        seen[cur] = 1
    return _induced(g, rows, list(seen))


def _dense_pattern(r, g, rows, k):
    """Grown a vertex at a time, the next one drawn by (its edges into the set) ** 4."""
    conn = np.zeros(g.n, np.int64)
    chosen = [int(r.integers(0, g.n))]
    edge = np.zeros(0, np.int64)
    while True:
        row = rows.row(chosen[-1])
        edge = np.concatenate([edge, row[conn[row] == 0]])
        conn[row] += 1
        conn[chosen] = -1
        edge = edge[conn[edge] > 0]
        if len(chosen) == k or edge.shape[0] == 0:
            break
        cum = np.cumsum(conn[edge] ** 4)
        chosen.append(int(edge[np.searchsorted(cum, r.random() * cum[-1], side="right")]))
    # as verts: the induced edges by sorted intersection (rows of hubs are long)
    verts = np.array(chosen)
    inv = np.full(g.n, -1)
    inv[verts] = np.arange(verts.shape[0])
    src, dst = [], []
    for i, v in enumerate(chosen):
        j = inv[rows.row(v)]
        j = j[j > i]
        src.append(np.full(j.shape[0], i))
        dst.append(j)
    return Graph(verts.shape[0], np.concatenate(src), np.concatenate(dst), g.vlabel[verts])


def _admit(E, tid, algo, make, lo, hi, tries, key="states"):
    """(pattern, its id) of the first of `tries` drawn ones whose search is in [lo, hi]; else of the
    largest below.  The search's state budget lies far above hi, so it decides nothing."""
    best = None
    for _ in range(tries):
        g = make()
        pid = E.load_pattern(g)
        res = E.count(tid, pid, check=False, algo=algo, state_budget=2 * max(hi, 1 << 20))
        size = res[key] if res["rc"] == 0 else hi + 1
        if size <= hi and (best is None or size > best[0]):
            if best is not None:
                sge.sge_unload_pattern(E.h, best[2])
            best = (size, g, pid)
            if size >= lo:
                break
        else:
            sge.sge_unload_pattern(E.h, pid)
    if best is None:   # every draw too large: one edge of the last, still a valid query
        g = Graph(2, [0], [1], g.vlabel[[g.src[0], g.dst[0]]], None if g.elabel is None else g.elabel[:1], g.directed)
        best = (0, g, E.load_pattern(g))
    return best[1], best[2]


# -------------------------------------------------------------------- cases
#: states of one pattern's search, per kind: what the searches kept lie between
STATES = {"dense": (100_000_000, 2_000_000_000), "network": (2_000, 10_000_000), "directed": (20_000, 20_000_000)}


def prepare(case, seed):
    r = np.random.default_rng([20170526, int(seed)])
    kind, algo = case["kind"], case["algo"]
    E = sge.Context(0)
    S = {"case": case, "E": E, "algo": algo}
    if kind in ("query", "list"):
        g = _random_graph(r, case["n"], case["degree"], case["labels"])
        rows = Rows(g)
        S["tid"] = E.load_target(g)
        lo, hi, key = (1, 1_000_000, "states") if kind == "query" else (6_000, 30_000, "matches")
        if kind == "list":
            S["room"] = np.zeros((hi, case["k"]), np.int32)   # the caller's array for the matches
        _, S["pid"] = _admit(E, S["tid"], algo, lambda: _walk_pattern(r, g, rows, case["k"]), lo, hi, 24, key)
        return S
    if kind == "molecules":
        targets = [_molecule(r) for _ in range(case["targets"])]
        rows = [Rows(g) for g in targets]
        S["tids"], S["pids"] = [], []
        for g in targets:
            S["tids"].append(E.load_target(g))
        for _ in range(case["pats"]):
            t = int(r.integers(0, len(targets)))
            k = min(int(4 * 16 ** r.random()), targets[t].n)   # 4 to 64 vertices, log-uniform
            S["pids"].append(E.load_pattern(_walk_pattern(r, targets[t], rows[t], k)))
        t, p = np.meshgrid(np.array(S["tids"], np.int32), np.array(S["pids"], np.int32), indexing="ij")
        S["tids"], S["pids"] = t.ravel(), p.ravel()
        return S
    if kind == "dense":
        g = _random_graph(r, case["n"], case["degree"], case["labels"])
    elif kind == "network":
        g = _network(r, case["n"], case["degree"], case["labels"])
    else:
        g = _random_graph(r, case["n"], case["degree"], case["labels"], True, case["elabels"])
    rows = Rows(g)
    tid = E.load_target(g)
    lo, hi = STATES[kind]
    pats, pids = [], []
    for i in range(case["pats"]):
        f = (i + 0.5) / case["pats"]   # sizes spread over the range, log-uniformly
        k = int(round(case["k_lo"] * (case["k_hi"] / case["k_lo"]) ** f))
        make = _walk_pattern if kind == "directed" else _dense_pattern
        p, pid = _admit(E, tid, algo, lambda: make(r, g, rows, k), lo, hi, 40 if kind == "dense" else 8)
        pats.append(p)
        pids.append(pid)
    if kind == "dense" and case["load"]:   # the job starts from host arrays
        S["target"], S["pats"] = g, pats
        sge.sge_unload_target(E.h, tid)
        for pid in pids:
            sge.sge_unload_pattern(E.h, pid)
    else:
        S["tids"], S["pids"] = np.full(len(pids), tid, np.int32), np.array(pids, np.int32)
    return S


def _columns(rows):
    return {k: rows[k] for k in ("matches", "states", "nodes", "hash")}


def run(S):
    E, case, algo = S["E"], S["case"], S["algo"]
    kind = case["kind"]
    if kind == "query":
        res = E.count(S["tid"], S["pid"], algo=algo)
        return np.array([res["matches"], res["states"], res["nodes"], res["hash"]], dtype=np.uint64)
    if kind == "list":
        res = E.enumerate(S["tid"], S["pid"], algo=algo)
        rows = res["match_list"]
        S["room"][:rows.shape[0], :rows.shape[1]] = rows
        return {"counters": np.array([res["matches"], res["states"], res["nodes"], res["hash"]], dtype=np.uint64),
                "match_list": S["room"]}
    if kind == "dense" and case["load"]:
        tid = E.load_target(S["target"])
        pids = [E.load_pattern(p) for p in S["pats"]]
        _, rows = E.count_batch([tid] * len(pids), pids, algo=algo)
        sge.sge_unload_target(E.h, tid)
        for p in pids:
            sge.sge_unload_pattern(E.h, p)
        return _columns(rows)
    if kind == "network" and case["serve"]:
        tickets = [E.serve_submit(int(t), int(p), algo=algo) for t, p in zip(S["tids"], S["pids"])]
        E.serve_drain()
        got = [E.serve_poll(t) for t in tickets]
        return {k: np.array([d[k] for d in got], dtype=np.uint64) for k in ("matches", "states", "nodes", "hash")}
    _, rows = E.count_batch(S["tids"], S["pids"], algo=algo)
    return _columns(rows)


def work(case):
    """Bytes: target and patterns in CSR with labels read once, results written once.  Operations: the
    (pattern vertex, target vertex) pairs that searches of this kind and size consider, one each."""
    kind = case["kind"]
    if kind == "molecules":
        pairs = case["targets"] * case["pats"]
        return {"bytes": case["targets"] * 260 * 27 + case["pats"] * 22 * 27 + pairs * 40, "flops": pairs * 500}
    arcs = case["n"] * case["degree"] * (2 if kind == "directed" else 1)
    graph = arcs * (8 if kind == "directed" else 4) + case["n"] * 8
    if kind in ("query", "list"):
        out = 15_000 * case["k"] * 4 if kind == "list" else 0
        return {"bytes": graph + case["k"] * 64 + 32 + out, "flops": 5_000 if kind == "query" else 200_000}
    k = math.sqrt(case["k_lo"] * case["k_hi"])
    per = {"dense": 400_000_000, "network": 1_000_000, "directed": 2_000_000}[kind]
    return {"bytes": int(graph + case["pats"] * (k * 64 + 32)), "flops": case["pats"] * per}


def exact(case, seed):
    """Nothing here is rounded: every output is a count, a 64-bit hash or a vertex id, compared for
    equality.  A search in plain numpy takes minutes for most of these cases."""
    return None
