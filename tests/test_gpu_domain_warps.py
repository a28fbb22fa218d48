"""The domain fixpoint of very many small pairs, one warp per pair over transposed domains:
patterns and targets at the edges of its 32-bit blocks and of its largest sizes, one to eight edge
classes (and nine, which it refuses), directed or not, pairs that lose a domain at the start, in a
sweep or to forward checking -- the counters are those of the block form and of the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from gen.graphs import Graph
from gpu_common import counters, engine

pytestmark = pytest.mark.gpu

BLOCKS = 2
PAIRS = 3000   # beyond the least batch that takes the warp form on any part with up to 375 SMs


def _target(seed, n, labels, directed, elabels):
    """A random tree with a tenth more edges: short rows, but for one vertex of degree n / 16."""
    r = np.random.default_rng(seed)
    par = np.array([int(r.integers(max(0, v - 9), v)) for v in range(1, n)])
    a, b = np.concatenate([par, r.integers(0, n, n // 10), np.zeros(n // 16, int)]), \
        np.concatenate([np.arange(1, n), r.integers(0, n, n // 10), r.integers(0, n, n // 16)])
    if directed:
        turn = r.integers(0, 2, a.shape[0]).astype(bool)
        a, b = np.where(turn, a, b), np.where(turn, b, a)
    else:
        a, b = np.minimum(a, b), np.maximum(a, b)
    key = np.unique((a * n + b)[a != b])
    return Graph(n, (key // n).astype(np.int32), (key % n).astype(np.int32),
                 r.integers(0, labels, n).astype(np.int32),
                 (r.integers(0, elabels, key.shape[0]) * 7 - 3).astype(np.int32) if elabels else None, directed)


def _pattern(seed, g, k, spoil):
    """k connected vertices of g with the edges among them; `spoil` changes one label."""
    r = np.random.default_rng(seed)
    nb = [[] for _ in range(g.n)]
    for s, d in zip(g.src.tolist(), g.dst.tolist()):
        nb[s].append(d)
        nb[d].append(s)
    verts = [int(r.integers(0, g.n))]
    while len(verts) < k:
        grow = sorted({y for x in verts for y in nb[x]} - set(verts))
        verts.append(grow[int(r.integers(0, len(grow)))])
    pos = {v: i for i, v in enumerate(verts)}
    keep = [e for e in range(g.src.shape[0]) if int(g.src[e]) in pos and int(g.dst[e]) in pos]
    lab = g.vlabel[verts].copy()
    if spoil:
        lab[int(r.integers(0, k))] = int(r.integers(0, 20))
    return Graph(k, np.array([pos[int(g.src[e])] for e in keep], np.int32),
                 np.array([pos[int(g.dst[e])] for e in keep], np.int32), lab,
                 None if g.elabel is None else g.elabel[keep], g.directed)


def _shifted(g):
    """g with its edge labels moved up by 3: the oracle marks a missing arc of a directed pattern by a
    negative label, and no counter depends on which labels they are."""
    return g if g.elabel is None else Graph(g.n, g.src, g.dst, g.vlabel, g.elabel + 3, g.directed)


@pytest.mark.parametrize("directed,elabels", [(False, 0), (False, 3), (False, 8), (False, 9), (True, 0), (True, 4),
                                              (True, 5)])
@pytest.mark.parametrize("nmax,kmax", [(64, 32), (512, 64), (513, 64), (512, 65)])
def test_warp_fixpoint(directed, elabels, nmax, kmax):
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    sizes = sorted({1, 2, 31, 32, 33, 64, 65, 200, nmax - 1, nmax})
    targets = [_target(7 * i + elabels, n, 20, directed, elabels) for i, n in enumerate(s for s in sizes if s <= nmax)]
    big = targets[-1]
    pats = [_pattern(31 * i + k, big if i % 2 or k > 60 else targets[-2], k, i % 3 == 1)
            for k in (1, 3, 8, 31, 32, 33, kmax - 1, kmax) if k <= kmax for i in range(3)]
    E = engine()
    tids, pids = [E.load_target(g) for g in targets], [E.load_pattern(p) for p in pats]
    try:
        r = np.random.default_rng(nmax + kmax)
        pick = [(int(r.integers(0, len(targets))), int(r.integers(0, len(pats)))) for _ in range(PAIRS)]
        a, b = [tids[t] for t, _ in pick], [pids[p] for _, p in pick]
        found = 0
        for algo in (1, 2, 3):
            rows = [counters(x) for x in E.count_batch(a, b, algo=algo)[1]]
            block = [counters(x) for x in E.count_batch(a, b, algo=algo, domain_fixpoint=BLOCKS)[1]]
            assert rows == block, algo
            some = sorted(set(pick))[algo::5]
            want = {x: counters(oracle.run(_shifted(targets[x[0]]), _shifted(pats[x[1]]), algo)) for x in some}
            assert all(rows[i] == want[x] for i, x in enumerate(pick) if x in want), algo
            found += sum(w[0] > 0 for w in want.values())
        assert found > 0
    finally:
        for p in pids:
            sge_unload_pattern(E.h, p)
        for t in tids:
            sge_unload_target(E.h, t)
