"""Donation in the CSR search when many warps start at once and most find nothing: a thousand heavy
frames for a device with several thousand warps, donors that look on every iteration and hand out
from one to 32 frames, undirected and directed, on targets with and without label runs, stopped and
resumed, and in the entry point whose queue has fewer cells than the device has warps."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu


def _target(seed, n, degree, directed):
    r = np.random.default_rng(seed)
    m = n * degree // (1 if directed else 2)
    a, b = r.integers(0, n, 2 * m), r.integers(0, n, 2 * m)
    lo, hi = (a, b) if directed else (np.minimum(a, b), np.maximum(a, b))
    key = np.unique((lo.astype(np.int64) * n + hi)[lo != hi])
    key = r.permutation(key)[:m]
    return Graph(n, (key // n).astype(np.int32), (key % n).astype(np.int32), np.zeros(n, np.int32), None, directed)


def _path(k, directed):
    i = np.arange(k - 1, dtype=np.int32)
    return Graph(k, i, i + 1, np.zeros(k, np.int32), None, directed)


@pytest.mark.parametrize("n,degree,k,directed", [(1201, 11, 5, False), (1201, 3, 10, False), (800, 12, 5, True)])
def test_heavy_frames_for_few_of_many_warps(n, degree, k, directed):
    from paper_1705_09358_gb300 import sge_count_noalloc, sge_unload_pattern, sge_unload_target
    g, p = _target(n + k, n, degree, directed), _path(k, directed)
    want = tuple(oracle.run(g, p, 0)[key] for key in ("matches", "states", "nodes", "hash"))
    assert want[1] > 5_000_000
    E = engine()
    tid, pid = E.load_target(g), E.load_pattern(p)
    try:
        for depth in (1, 2):
            for opts in ({}, {"steal_granularity": 1}, {"steal_granularity": 32, "donate_every_iters": 1},
                         {"donate_every_iters": 1, "blocks_per_sm": 1}, {"donate_every_us": 1}):
                res = E.count(tid, pid, kernel=1, split_depth=depth, **opts)
                assert counters(res) == want, (depth, opts)
                assert res["donations"] > 0
        # stopped before the end, then resumed with the frames that are left: all start at once
        rc, rows, blob = E.count_batch_ckpt([tid], [pid], kernel=1, split_depth=1, state_budget=want[1] // 4)
        assert rc == -4 and blob is not None
        for _ in range(200):
            rc, rows, blob = E.resume(blob, kernel=1, donate_every_iters=1, state_budget=want[1] // 3)
            if blob is None:
                break
        assert rc == 0 and counters(rows[0]) == want
        if not directed:
            import torch
            from test_zz_no_alloc import _device_csr
            d = _device_csr(g)
            rc, got = sge_count_noalloc(g.n, d["rowptr"].data_ptr(), d["col"].data_ptr(), d["vlabel"].data_ptr(), 0, p,
                                        stream=torch.cuda.current_stream())
            assert rc == 0 and counters(got) == want
    finally:
        sge_unload_pattern(E.h, pid)
        sge_unload_target(E.h, tid)


def test_default_cadence_costs_no_more_than_a_wide_one():
    """Looking for idle warps must not be what the search spends its time on: the default against
    one look in 64 iterations, alternating (on directed patterns from few frames a look at
    every iteration took 2.2 times as long)."""
    from time import perf_counter
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    g, p = _target(3, 3001, 10, True), _path(5, True)
    E = engine()
    tid, pid = E.load_target(g), E.load_pattern(p)
    try:
        times = {0: [], 64: []}
        for _ in range(12):
            for iters in times:
                t0 = perf_counter()
                E.count(tid, pid, kernel=1, split_depth=1, donate_every_iters=iters)
                times[iters].append(perf_counter() - t0)
        best = {i: sorted(t)[len(t) // 4] for i, t in times.items()}
        assert best[0] < 1.5 * best[64], best
    finally:
        sge_unload_pattern(E.h, pid)
        sge_unload_target(E.h, tid)


def test_a_search_from_one_frame_spreads_as_fast_as_a_batched_call():
    """sge_count_noalloc starts from the root alone: sharing that out must not make it several times
    as long as the batched call on the same kernel from a split of depth 1 (2.5 times when donors
    handed out two frames in 1,024 iterations)."""
    from time import perf_counter
    import torch
    from paper_1705_09358_gb300 import sge_count_noalloc, sge_unload_pattern, sge_unload_target
    from test_zz_no_alloc import _device_csr
    g, p = _target(5, 2001, 40, False), _path(4, False)
    E = engine()
    tid, pid = E.load_target(g), E.load_pattern(p)
    d = _device_csr(g)
    try:
        times = {"batched": [], "noalloc": []}
        for _ in range(12):
            t0 = perf_counter()
            want = E.count(tid, pid, kernel=1, split_depth=1)
            t1 = perf_counter()
            rc, got = sge_count_noalloc(g.n, d["rowptr"].data_ptr(), d["col"].data_ptr(), d["vlabel"].data_ptr(), 0, p,
                                        stream=torch.cuda.current_stream())
            t2 = perf_counter()
            assert rc == 0 and counters(got) == counters(want)
            times["batched"].append(t1 - t0)
            times["noalloc"].append(t2 - t1)
        best = {k: sorted(t)[len(t) // 4] for k, t in times.items()}
        assert best["noalloc"] < 2.5 * best["batched"], best
    finally:
        sge_unload_pattern(E.h, pid)
        sge_unload_target(E.h, tid)


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("hub", [63, 64, 65, 500, 1500])
def test_a_hub_with_one_level_below_is_shared(hub, directed):
    """Frames that start on the last position but one: the range of a long one is handed out in
    halves (nothing was, and one warp searched below a hub alone)."""
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    n = hub + 200
    r = np.random.default_rng(hub)
    # vertex 0 to `hub` others, which form a dense graph with the rest
    a, b = r.integers(1, n, 40 * n), r.integers(1, n, 40 * n)
    key = np.unique((np.minimum(a, b).astype(np.int64) * n + np.maximum(a, b))[a != b])
    key = np.concatenate([np.arange(1, hub + 1, dtype=np.int64), key])
    lab = np.zeros(n, np.int32)
    lab[0] = 1
    g = Graph(n, (key // n).astype(np.int32), (key % n).astype(np.int32), lab, None, directed)
    p = Graph(3, np.array([0, 0], np.int32), np.array([1, 2], np.int32), np.array([1, 0, 0], np.int32), None, directed)
    E = engine()
    tid, pid = E.load_target(g), E.load_pattern(p)
    try:
        for algo in (0, 1):
            want = tuple(oracle.run(g, p, algo)[key] for key in ("matches", "states", "nodes", "hash"))
            for copies in (1, 5):
                given = 0
                for opts in ({"split_depth": 1}, {"split_depth": 1, "donate_every_iters": 1}, {"state_budget": 1 << 60}):
                    rc, rows = E.count_batch([tid] * copies, [pid] * copies, algo=algo, kernel=1, tuned=False, **opts)
                    assert [counters(x) for x in rows] == [want] * copies, (algo, opts)
                    given += int(rows["donations"][0])
                assert hub < 500 or given > 0, (algo, copies)
    finally:
        sge_unload_pattern(E.h, pid)
        sge_unload_target(E.h, tid)
