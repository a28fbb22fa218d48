"""Serving RI-DS queries while another group's long search runs: a search that occupies one block of
the device for a second must not hold up the domains of queries served beside it."""
from __future__ import annotations

import time

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu


def _target(n, m, seed):
    """A random graph of label 0 with one vertex of label 1, joined to 40 others."""
    r = np.random.default_rng(seed)
    a, b = r.integers(1, n, 2 * m), r.integers(1, n, 2 * m)
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    key = np.unique((lo.astype(np.int64) * n + hi)[lo != hi])
    key = np.concatenate([np.arange(1, 41, dtype=np.int64), r.permutation(key)[:m]])
    lab = np.zeros(n, np.int32)
    lab[0] = 1
    return Graph(n, (key // n).astype(np.int32), (key % n).astype(np.int32), lab, None, False)


def _star_path(k):
    """A star whose centre of label 1 has 8 leaves, one of them the end of a path of k."""
    src = [0] * 8 + [1] + list(range(9, 8 + k))
    dst = list(range(1, 9)) + list(range(9, 9 + k))
    lab = np.zeros(9 + k, np.int32)
    lab[0] = 1
    return Graph(9 + k, np.array(src, np.int32), np.array(dst, np.int32), lab, None, False)


def test_domains_beside_a_long_search():
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    E = engine()
    g = _target(3000, 60000, 3)
    long_pattern = _star_path(12)
    short = Graph(4, np.array([0, 1, 2], np.int32), np.array([1, 2, 3], np.int32), np.array([1, 0, 0, 0], np.int32),
                  None, False)
    tid = E.load_target(g)
    pl, ps = E.load_pattern(long_pattern), E.load_pattern(short)
    try:
        want = tuple(oracle.run(g, short, 3)[k] for k in ("matches", "states", "nodes", "hash"))
        # one root candidate, one frame, nothing handed on: one warp searches until the limit
        slow = dict(algo=0, kernel=1, split_depth=1, no_donation=1, time_limit_ms=700)
        waits = []
        for _ in range(5):   # (a worker's first group beside it may wait for device memory to be mapped)
            ticket = E.serve_submit(tid, pl, **slow)
            time.sleep(0.1)
            t0 = time.perf_counter()
            tickets = [E.serve_submit(tid, ps, algo=3) for _ in range(3)]
            rows = []
            while len(rows) < 3 and time.perf_counter() - t0 < 5.0:
                for t in list(tickets):
                    d = E.serve_poll(t)
                    if d is not None:
                        rows.append(d)
                        tickets.remove(t)
            waits.append(time.perf_counter() - t0)
            E.serve_drain()
            assert [counters(d) for d in rows] == [want] * 3
            d = E.serve_poll(ticket)
            assert d["status"] == -5 and d["search_kernel_ms"] > 600   # (it did run that long)
        assert min(waits) < 0.2, waits
    finally:
        sge_unload_pattern(E.h, pl)
        sge_unload_pattern(E.h, ps)
        sge_unload_target(E.h, tid)
