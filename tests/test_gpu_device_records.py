"""Huge plain RI batches, whose job records and root frames the device puts together from the
distinct graphs' tables: every counter is that of the same pairs in calls too small for it, and of
the oracle -- for patterns that are larger than the target, disconnected or one vertex, targets
without edges, roots cut into ranges, shards, budgets and calls with the general path between."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu

FEW, MANY = 4095, 4096   # the last batch of host records, the first of device records


def _graph(seed, n, m, labels, directed, elabels):
    r = np.random.default_rng(seed)
    a, b = r.integers(0, n, 4 * m + 1), r.integers(0, n, 4 * m + 1)
    if not directed:
        a, b = np.minimum(a, b), np.maximum(a, b)
    key = r.permutation(np.unique((a * n + b)[a != b]))[:m]
    src, dst = np.sort(key) // n, np.sort(key) % n
    return Graph(n, src.astype(np.int32), dst.astype(np.int32), r.integers(0, labels, n).astype(np.int32),
                 r.integers(0, 2, src.shape[0]).astype(np.int32) if elabels else None, directed)


@pytest.mark.parametrize("directed,elabels", [(False, False), (False, True), (True, False), (True, True)])
def test_device_built_records(directed, elabels):
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    # (mean rows below 4: no label runs; 3,000 vertices: roots cut into ranges)
    targets = [_graph(100 + i, n, m, 3, directed, elabels) for i, (n, m) in
               enumerate([(1, 0), (2, 1), (9, 12), (33, 50), (64, 90), (150, 200), (3000, 4000)])]
    pats = [_graph(200 + i, n, m, 3, directed, elabels) for i, (n, m) in
            enumerate([(1, 0), (2, 1), (2, 0), (3, 2), (4, 3), (5, 4), (6, 3), (12, 14)])]
    E = engine()
    tids = [E.load_target(g) for g in targets]
    for _ in range(3):   # ids with gaps: some loaded graphs are in no pair
        tids.append(E.load_target(targets[2]))
    pids = [E.load_pattern(p) for p in pats]
    try:
        # patterns 2 and 6 on the largest target are left out: too many matches for the oracle
        legal = [(t, p) for t in range(len(targets)) for p in range(len(pats))
                 if (t < 5 or p not in (2, 6)) and not (t == 6 and p == 7)]
        want = {x: counters(oracle.run(targets[x[0]], pats[x[1]], 0)) for x in legal}
        assert any(w[0] > 0 for w in want.values())
        r = np.random.default_rng(1)
        for count in (FEW, MANY, MANY + 33, 20000):
            pick = [legal[i] for i in r.integers(0, len(legal), count)]
            a, b = [tids[t] for t, _ in pick], [pids[p] for _, p in pick]
            for opts in ({}, {"frontier_kib": 1}, {"no_donation": 1}, {"split_depth": 1}):
                rc, rows = E.count_batch(a, b, kernel=1, **opts)
                assert [counters(x) for x in rows] == [want[x] for x in pick], (count, opts)
            got = [counters(x) for x in E.count_batch(a, b)[1]]   # the kernel left to the engine
            assert got == [want[x] for x in pick], count
        total = np.zeros((len(pick), 3), np.uint64)
        for s in range(3):
            rc, rows = E.count_batch(a, b, kernel=1, shard_count=3, shard_index=s)
            total += np.array([[x["matches"], x["states"], x["nodes"]] for x in rows], np.uint64)
        assert [tuple(int(v) for v in x) for x in total] == [want[x][:3] for x in pick]
        rc, rows = E.count_batch(a, b, kernel=1, state_budget=1 << 50)
        assert rc == 0 and [counters(x) for x in rows] == [want[x] for x in pick]
    finally:
        for p in pids:
            sge_unload_pattern(E.h, p)
        for t in tids:
            sge_unload_target(E.h, t)
