"""The whole-device domain fixpoint that small RI-DS calls use: the same counters as the sweeps under
the host loop and the oracle, for one pair and for several, empty domains and chains of forward
checking among them, on either side of the adjacency-bitset limit, directed and edge-labelled."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine
from test_gpu_label_runs import _graph, _pattern

pytestmark = pytest.mark.gpu

SWEEPS = 1


def _chain(n):
    """A path whose labels force one vertex after another to a singleton domain."""
    src = np.arange(n - 1, dtype=np.int32)
    return Graph(n, src, src + 1, np.array([7] + [1] * (n - 1), np.int32), None, False)


@pytest.mark.parametrize("n,m,labels,hubs,directed,elabels", [
    (64, 300, 2, 0, False, 0), (65, 300, 2, 0, True, 2), (900, 4000, 3, 1, False, 0), (900, 2000, 3, 1, True, 0),
    (16384, 30000, 30, 0, False, 1), (16385, 40000, 30, 1, False, 0), (1, 0, 1, 0, False, 0)])
def test_few_pairs(n, m, labels, hubs, directed, elabels):
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    g = _graph(3 * n + m, n, m, labels, hubs, directed, elabels) if m else Graph(
        1, np.zeros(0, np.int32), np.zeros(0, np.int32), np.array([4], np.int32), None, False)
    pats = [_pattern(s, g, 2 + s % 3, extra_label=s == 4) for s in range(9)] if m else [
        Graph(1, g.src, g.dst, np.array([x], np.int32), None, False) for x in (4, 5)]
    if not directed and not elabels and m:
        pats += [_chain(2), _chain(5)]
    E = engine()
    tid = E.load_target(g)
    pids = [E.load_pattern(p) for p in pats]
    try:
        for algo in (1, 2, 3):
            want = [tuple(oracle.run(g, p, algo)[k] for k in ("matches", "states", "nodes", "hash")) for p in pats]
            for some in ([0], list(range(len(pids))), [i % len(pids) for i in range(31)]):
                for mode in (0, SWEEPS):
                    rc, rows = E.count_batch([tid] * len(some), [pids[i] for i in some], algo=algo,
                                             domain_fixpoint=mode)
                    assert [counters(r) for r in rows] == [want[i] for i in some], (algo, some, mode)
    finally:
        for p in pids:
            sge_unload_pattern(E.h, p)
        sge_unload_target(E.h, tid)


@pytest.mark.parametrize("k", [2, 3, 31, 100])
def test_forward_checking_walks_a_path(k):
    """Pattern and target are one path with a distinct end label: each singleton fixes the next."""
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    g, p = _chain(k), _chain(k)
    E = engine()
    tid, pid = E.load_target(g), E.load_pattern(p)
    try:
        for algo in (1, 3):
            want = tuple(oracle.run(g, p, algo)[key] for key in ("matches", "states", "nodes", "hash"))
            assert want[0] == 1
            for mode in (0, SWEEPS):
                assert counters(E.count(tid, pid, algo=algo, domain_fixpoint=mode)) == want
    finally:
        sge_unload_pattern(E.h, pid)
        sge_unload_target(E.h, tid)
