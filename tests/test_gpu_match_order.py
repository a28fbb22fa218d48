"""Listed matches come sorted by the images of pattern vertices 0, 1, ..., at the sizes where the sort's
tiles, its merge passes and the first buffer's room end."""
from __future__ import annotations

import itertools

import numpy as np
import pytest

from gen.graphs import Graph
from gpu_common import engine

pytestmark = pytest.mark.gpu


def _complete(n):
    a, b = np.triu_indices(n, 1)
    return Graph(n, a.astype(np.int32), b.astype(np.int32), np.zeros(n, np.int32), None, False)


def _edgeless(n):
    none = np.zeros(0, np.int32)
    return Graph(n, none, none, np.zeros(n, np.int32), None, False)


def _list(target, pattern, **opts):
    from paper_1705_09358_gb300 import sge_unload_pattern, sge_unload_target
    E = engine()
    tid, pid = E.load_target(target), E.load_pattern(pattern)
    try:
        return E.enumerate(tid, pid, **opts)
    finally:
        sge_unload_pattern(E.h, pid)
        sge_unload_target(E.h, tid)


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 2049, 65535, 65536, 65537, 131073])
def test_single_vertices(n):
    got = _list(_edgeless(n), _edgeless(1))
    assert got["matches"] == n and np.array_equal(got["match_list"][:, 0], np.arange(n))


@pytest.mark.parametrize("n,k", [(2, 2), (32, 2), (33, 2), (256, 2), (257, 2), (41, 3), (42, 3), (16, 4), (17, 4), (7, 6), (9, 6)])
@pytest.mark.parametrize("algo", [0, 3])
def test_complete_graphs(n, k, algo):
    """K_k in K_n: every ordered choice of k vertices, in ascending order."""
    got = _list(_complete(n), _complete(k), algo=algo)
    want = np.array(list(itertools.permutations(range(n), k)), dtype=np.int32)
    assert got["matches"] == want.shape[0] and np.array_equal(got["match_list"], want)


def test_no_match():
    got = _list(_edgeless(5), _complete(2))
    assert got["matches"] == 0 and got["match_list"].shape == (0, 0)
