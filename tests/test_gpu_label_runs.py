"""Label runs (rows regrouped by neighbour label): a node's candidates are the shortest run
among its earlier neighbours' rows, whichever that is, and everything that counts or cuts
candidate lists -- states, range frames, donations, checkpoints -- still follows the parent's row."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu

BUDGET = -4


def _graph(seed, n, m, labels, hubs=0, directed=False, elabels=0, absent=0):
    """Random edges plus `hubs` vertices joined to every other one; labels 1000 + 7 * index."""
    r = np.random.default_rng(seed)
    a, b = r.integers(0, n, 2 * m), r.integers(0, n, 2 * m)
    for h in range(hubs):
        others = np.delete(np.arange(n), h)
        a, b = np.concatenate([a, np.full(n - 1, h)]), np.concatenate([b, others])
    if not directed:
        a, b = np.minimum(a, b), np.maximum(a, b)
    key = np.unique((a * n + b)[a != b])
    if hubs == 0:
        key = np.sort(r.permutation(key)[:m])
    src, dst = key // n, key % n
    el = r.integers(0, elabels + 1, key.shape[0]) if elabels else None
    return Graph(n, src.astype(np.int32), dst.astype(np.int32), (1000 + 7 * r.integers(0, labels, n)).astype(np.int32),
                 None if el is None else el.astype(np.int32), directed)


def _pattern(seed, g, k, extra_label=False):
    """A connected k-vertex subgraph grown from a random vertex (hub or not)."""
    r = np.random.default_rng(seed)
    nb = [[] for _ in range(g.n)]
    for e in range(g.src.shape[0]):
        nb[g.src[e]].append(int(g.dst[e]))
        nb[g.dst[e]].append(int(g.src[e]))
    while True:
        verts = [int(r.integers(0, g.n))]
        while len(verts) < k:
            grow = sorted({y for x in verts for y in nb[x]} - set(verts))
            if not grow:
                break
            verts.append(grow[int(r.integers(0, len(grow)))])
        if len(verts) == k:
            break
    pos = {v: i for i, v in enumerate(verts)}
    keep = [e for e in range(g.src.shape[0]) if int(g.src[e]) in pos and int(g.dst[e]) in pos]
    lab = g.vlabel[verts].copy()
    if extra_label:
        lab[-1] = 5   # a label the target does not have
    return Graph(k, np.array([pos[int(g.src[e])] for e in keep], np.int32),
                 np.array([pos[int(g.dst[e])] for e in keep], np.int32), lab,
                 None if g.elabel is None else g.elabel[keep], g.directed)


def _drain(E, blob, **opts):
    for _ in range(500):
        rc, rows, blob = E.resume(blob, **opts)
        if blob is None:
            return rows
    raise AssertionError("the search did not finish")


CASES = [
    # n, m, labels, hubs, directed, edge labels
    (400, 799, 3, 0, False, 0),      # mean row just below the limit: no runs
    (400, 800, 3, 0, False, 0),      # ... and just at it
    (130, 1300, 1, 0, False, 0),     # one label: a run is the row
    (700, 5000, 64, 0, False, 0),    # most runs empty or one entry
    (2300, 3000, 2, 2, False, 0),    # hub runs of about 1,150 entries: cut into ranges
    (2300, 3000, 2, 2, False, 2),    # ... with edge labels
    (17000, 34000, 4, 1, False, 0),  # above the adjacency-bitset limit: hub rows and searches
    (300, 2000, 3, 0, True, 0),      # directed
    (2300, 2500, 2, 2, True, 2),     # directed hubs with edge labels
]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("algo", [0, 3])
def test_counters_follow_the_oracle(case, algo):
    n, m, labels, hubs, directed, elabels = case
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    g = _graph(n + m, n, m, labels, hubs, directed, elabels)
    ks = (2, 3) if hubs else (2, 3, 4, 5)
    pats = [_pattern(17 * k + s, g, k, extra_label=s == 3) for k in ks for s in range(4)]
    want = [tuple(oracle.run(g, p, algo)[key] for key in ("matches", "states", "nodes", "hash")) for p in pats]
    E = engine()
    tid = E.load_target(g)
    pids = [E.load_pattern(p) for p in pats]
    try:
        kernels = [1] if directed or elabels or n > 8192 else [1, 2]
        for kernel in kernels:
            for opts in ({}, {"split_depth": 1}, {"split_depth": 1, "frontier_kib": 4}, {"no_donation": 1}):
                rc, rows = E.count_batch([tid] * len(pids), pids, algo=algo, kernel=kernel, **opts)
                assert [counters(r) for r in rows] == want, (kernel, opts)
            total = np.zeros((len(pats), 4), np.uint64)
            for shard in range(2):
                rc, rows = E.count_batch([tid] * len(pids), pids, algo=algo, kernel=kernel, shard_index=shard,
                                         shard_count=2)
                total += np.array([counters(r) for r in rows], np.uint64)
            assert [tuple(int(x) for x in r) for r in total] == want, (kernel, "shards")
            # stopped early, with ranges of runs in the frontier, the queue and the warps' hands
            budget = max(w[1] for w in want) // 5 + 1
            for depth in (1, 2):
                rc, rows, blob = E.count_batch_ckpt([tid] * len(pids), pids, algo=algo, kernel=kernel,
                                                    state_budget=budget, split_depth=depth, frames_per_warp=1)
                assert rc in (0, BUDGET)
                if blob is not None:
                    other = kernels[-1] if kernel == 1 else 1
                    rows = _drain(E, blob, kernel=other, state_budget=2 * budget)
                assert [counters(r) for r in rows] == want, (kernel, "resumed", depth)
    finally:
        for p in pids:
            sge_unload_pattern(E.h, p)
        sge_unload_target(E.h, tid)
