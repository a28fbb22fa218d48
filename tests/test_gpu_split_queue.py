"""The queue of the split's end without barriers, when it is full before the arena is: it has one
entry per 64 ints of the frontier buffer, and a frame here takes 6 to 9.  What is left goes to the
search, counted once."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("kib", [2, 40, 200, 1000])
def test_full_queue(kib, directed):
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    r = np.random.default_rng(5)
    n = 1200
    key = np.unique(r.integers(0, n, 24000) * n + r.integers(0, n, 24000))
    src, dst = key // n, key % n
    keep = src < dst
    # few roots, of label 0, then a burst
    g = Graph(n, src[keep].astype(np.int32), dst[keep].astype(np.int32), (r.integers(0, 200, n) > 0).astype(np.int32),
              None, directed)
    # (the vertex of label 0 has the most neighbours, so it comes first)
    a, b = np.array([0, 0, 0, 3, 4], np.int32), np.array([1, 2, 3, 4, 5], np.int32)
    p = Graph(6, a, b, np.array([0, 1, 1, 1, 1, 1], np.int32), None, directed)
    E = engine()
    tid, pid = E.load_target(g), E.load_pattern(p)
    try:
        for algo in (0, 3):
            want = tuple(oracle.run(g, p, algo)[k] for k in ("matches", "states", "nodes", "hash"))
            assert want[0] > 5000
            for copies in (1, 7):
                rc, rows = E.count_batch([tid] * copies, [pid] * copies, algo=algo, kernel=1, frontier_kib=kib)
                assert [counters(x) for x in rows] == [want] * copies, (algo, copies)
    finally:
        sge_unload_pattern(E.h, pid)
        sge_unload_target(E.h, tid)
