"""Device blocks that a call can do without: when one is not to be had, the call takes its other
way and gives the same results.  SGE_BLOCK_MAX makes larger blocks count as not to be had."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine
from test_gpu_label_runs import _graph, _pattern

pytestmark = pytest.mark.gpu

KEYS = ("matches", "states", "nodes", "hash")


@pytest.fixture
def fresh():
    """A context of its own: no block is there from earlier calls."""
    import paper_1705_09358_gb300 as sge
    engine()
    with sge.Context(0) as E:
        yield E


@pytest.mark.parametrize("directed", [False, True])
def test_target_without_room_for_label_runs(fresh, monkeypatch, directed):
    g = _graph(7, 2000, 12000, 150, 1, directed, 2 if directed else 0)
    pats = [_pattern(s, g, 3 + s % 3) for s in range(6)]
    table = 2000 * 151 * 4                      # the runs' table alone, per direction
    monkeypatch.setenv("SGE_BLOCK_MAX", str(table + 20_000))
    tid = fresh.load_target(g)
    monkeypatch.delenv("SGE_BLOCK_MAX")
    pids = [fresh.load_pattern(p) for p in pats]
    for algo in range(4):
        want = [tuple(oracle.run(g, p, algo)[k] for k in KEYS) for p in pats]
        for kernel in (0, 1):
            rc, rows = fresh.count_batch([tid] * len(pids), pids, algo=algo, kernel=kernel)
            assert [counters(r) for r in rows] == want, (algo, kernel)


# the largest block that a call below cannot do without, the list of what the split leaves: 36.7 MB
ROOM = 37_500_000


def test_few_pairs_without_room_for_the_domain_slots(fresh, monkeypatch):
    """12 bytes for every vertex that may carry a pattern vertex's label, here 43 MB: the sweeps,
    which list the candidates there are, take the call."""
    n = 20_000
    g = _graph(11, n, 4 * n, 1)
    pats = [_pattern(s, g, 3) for s in range(3)]
    tid, pids = fresh.load_target(g), [fresh.load_pattern(p) for p in pats] * 20
    assert 12 * n * 3 * len(pids) > ROOM
    for algo in (1, 3):
        want = [tuple(oracle.run(g, p, algo)[k] for k in KEYS) for p in pats] * 20
        launches = {}
        for room in (ROOM, None):
            if room:
                monkeypatch.setenv("SGE_BLOCK_MAX", str(room))
            else:
                monkeypatch.delenv("SGE_BLOCK_MAX")
            rc, rows = fresh.count_batch([tid] * len(pids), pids, algo=algo, tuned=False, frontier_kib=1024)
            assert [counters(r) for r in rows] == want, (algo, room)
            launches[room] = int(rows["launches"][0])
        if algo == 1:   # (the second variant finds the slots' block there)
            assert launches[ROOM] > launches[None]


def test_split_without_room_for_its_queue(fresh, monkeypatch):
    """The levels then go on to the end one by one; the call after it has the queue again."""
    from test_gpu_split_async import _broom, _pattern as _handle
    handles = [2, 17, 60, 125]
    g = _broom(handles, 30)
    starts = np.cumsum([0] + [h + 90 for h in handles[:-1]])
    pats = [_handle(g, h, int(s)) for h, s in zip(handles, starts)]
    tid, pids = fresh.load_target(g), [fresh.load_pattern(p) for p in pats]
    want = [tuple(oracle.run(g, p, 0)[k] for k in KEYS) for p in pats] * 5
    for room in (ROOM // 2, None, ROOM // 2, None):   # (18.7 MB: the entries fit, the list does not)
        if room:
            monkeypatch.setenv("SGE_BLOCK_MAX", str(room))
        else:
            monkeypatch.delenv("SGE_BLOCK_MAX")
        for kib in (1024, 16):
            rc, rows = fresh.count_batch([tid] * 20, pids * 5, kernel=1, frontier_kib=kib)
            assert [counters(r) for r in rows] == want, (room, kib)


def test_listing_without_room_to_sort_on_the_device(fresh, monkeypatch):
    """24 bytes a match to sort, 38.4 MB here, against 8 to list: then the host sorts."""
    n, m = 50_000, 800_000
    r = np.random.default_rng(2)
    key = np.unique(r.integers(0, n, 3 * m) * n + r.integers(0, n, 3 * m))
    src, dst = key // n, key % n
    keep = r.permutation(np.flatnonzero(src < dst))[:m]
    g = Graph(n, src[keep].astype(np.int32), dst[keep].astype(np.int32), np.zeros(n, np.int32), None, False)
    edge = Graph(2, np.array([0], np.int32), np.array([1], np.int32), np.zeros(2, np.int32), None, False)
    tid, pid = fresh.load_target(g), fresh.load_pattern(edge)
    both = np.concatenate([np.stack([g.src, g.dst], 1), np.stack([g.dst, g.src], 1)])
    want = both[np.lexsort((both[:, 1], both[:, 0]))]
    launches = {}
    for room in (ROOM, None, None):
        if room:
            monkeypatch.setenv("SGE_BLOCK_MAX", str(room))
        else:
            monkeypatch.delenv("SGE_BLOCK_MAX", raising=False)
        got = fresh.enumerate(tid, pid, frontier_kib=4096)
        assert got["matches"] == 2 * m and np.array_equal(got["match_list"], want)
        launches[room] = got["launches"]
    assert launches[ROOM] < launches[None]
