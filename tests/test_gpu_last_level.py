"""The last level of the breadth-first split cuts lists of label runs into parts of 256 entries, the
levels before it into parts of 1,024: lists on either side of both, on the last position and on the
one before it, in batches wide and narrow."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu


def _target(lists, directed):
    """Hubs (label 1), each with a list of its length of leaves (labels 2 and 3 alternating); the
    leaves joined in a ring of degree 8, so that rows are long enough for label runs."""
    lab, edges = [], []
    for x in lists:
        hub = len(lab)
        lab += [1] + [2 + i % 2 for i in range(2 * x)]
        edges += [(hub, hub + 1 + i) for i in range(2 * x)]
    leaves = np.flatnonzero(np.array(lab) != 1)
    for d in range(1, 5):
        edges += [(int(a), int(b)) for a, b in zip(leaves, np.roll(leaves, d))]
    e = sorted({(min(p), max(p)) for p in edges if p[0] != p[1]})
    s, d = np.array(e, np.int32).T
    return Graph(len(lab), s, d, np.array(lab, np.int32), None, directed)


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("x", [255, 256, 257, 512, 513, 1024, 1025])
def test_parts_of_long_lists(x, directed):
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    g = _target([x, 3, x // 2], directed)
    star = Graph(3, np.array([0, 0], np.int32), np.array([1, 2], np.int32), np.array([1, 2, 3], np.int32), None, directed)
    edge = Graph(2, np.array([0], np.int32), np.array([1], np.int32), np.array([1, 2], np.int32), None, directed)
    tail = Graph(4, np.array([0, 0, 0], np.int32), np.array([1, 2, 3], np.int32), np.array([1, 2, 3, 9], np.int32), None,
                 directed)   # (a label the target lacks on the last position)
    E = engine()
    tid = E.load_target(g)
    pids = [E.load_pattern(p) for p in (star, edge, tail)]
    try:
        for algo in (0, 1):
            want = [tuple(oracle.run(g, p, algo)[k] for k in ("matches", "states", "nodes", "hash")) for p in (star, edge, tail)]
            assert want[1][0] >= x
            for copies in (1, 60):
                for opts in ({}, {"no_donation": 1}, {"frontier_kib": 64}, {"split_depth": 2}):
                    rc, rows = E.count_batch([tid] * 3 * copies, pids * copies, algo=algo, kernel=1, tuned=False, **opts)
                    assert [counters(r) for r in rows] == want * copies, (algo, copies, opts)
    finally:
        for p in pids:
            sge_unload_pattern(E.h, p)
        sge_unload_target(E.h, tid)
