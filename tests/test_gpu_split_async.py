"""The end of the breadth-first split without barriers: searches that stay narrow for many
levels, then burst, at several depths in one batch, with arenas that hold everything, run out in
the burst, or hold nothing -- the counters are those of the oracle every time."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu


def _broom(handles, leaves, directed=False, elabels=False):
    """Paths of labels 0, 1, .. (one per handle length), the last vertex of each joined to
    `leaves` vertices of label 99 with two neighbours of label 98 each."""
    lab, src, dst = [], [], []
    for h in handles:
        base = len(lab)
        lab += [1000 * h + i for i in range(h)]
        src += range(base, base + h - 1)
        dst += range(base + 1, base + h)
        for _ in range(leaves):
            leaf = len(lab)
            lab += [99, 98, 98]
            src += [base + h - 1, leaf, leaf]
            dst += [leaf, leaf + 1, leaf + 2]
    # enough extra edges among the label-98 vertices that rows are long enough for label runs
    ends = [v for v, x in enumerate(lab) if x == 98]
    r = np.random.default_rng(len(ends))
    have = set(zip(src, dst)) | set(zip(dst, src))
    while len(src) < 2.2 * len(lab):
        a, b = (int(x) for x in r.choice(ends, 2, replace=False))
        if (a, b) not in have and (b, a) not in have:
            have.add((a, b))
            src.append(a)
            dst.append(b)
    s, d = np.array(src, np.int32), np.array(dst, np.int32)
    return Graph(len(lab), s, d, np.array(lab, np.int32), (1 + (s + d) % 2).astype(np.int32) if elabels else None,
                 directed)


def _pattern(g, h, start):
    """The handle of length h, two of its leaves, and one end of the first."""
    verts = list(range(start, start + h)) + [start + h, start + h + 1, start + h + 3]
    pos = {v: i for i, v in enumerate(verts)}
    keep = [e for e in range(g.src.shape[0]) if int(g.src[e]) in pos and int(g.dst[e]) in pos]
    return Graph(len(verts), np.array([pos[int(g.src[e])] for e in keep], np.int32),
                 np.array([pos[int(g.dst[e])] for e in keep], np.int32), g.vlabel[verts],
                 None if g.elabel is None else g.elabel[keep], g.directed)


@pytest.mark.parametrize("directed,elabels", [(False, False), (False, True), (True, True)])
@pytest.mark.parametrize("leaves", [7, 70])
def test_narrow_searches_that_burst(directed, elabels, leaves):
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    handles = [2, 3, 17, 40, 60, 100, 125]
    g = _broom(handles, leaves, directed, elabels)
    starts = np.cumsum([0] + [h + 3 * leaves for h in handles[:-1]])
    pats = [_pattern(g, h, int(s)) for h, s in zip(handles, starts)]
    assert max(p.n for p in pats) == 128
    E = engine()
    tid = E.load_target(g)
    pids = [E.load_pattern(p) for p in pats]
    try:
        for algo in (0, 1):
            want = [tuple(oracle.run(g, p, algo)[k] for k in ("matches", "states", "nodes", "hash")) for p in pats]
            assert min(w[0] for w in want) >= leaves
            for copies in (1, 40):
                for kib in (0, 1, 16, 100, 600, 4000):
                    rc, rows = E.count_batch([tid] * (len(pids) * copies), pids * copies, algo=algo, kernel=1,
                                             frontier_kib=kib)
                    assert [counters(r) for r in rows] == want * copies, (algo, copies, kib)
    finally:
        for p in pids:
            sge_unload_pattern(E.h, p)
        sge_unload_target(E.h, tid)
