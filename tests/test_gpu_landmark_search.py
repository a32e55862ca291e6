"""Landmark searches of deep graphs, a block from each landmark: the
distances equal breadth-first search where the search could go wrong
(vertices of 63 to 65 and of many arcs, vertices no landmark reaches, sizes
around a word of its bits, searches that stop within the levels run before
it), and the spread landmarks keep their definition."""
from __future__ import annotations

import numpy as np
import pytest

import pspc_inputs as P
from tests.test_gpu_landmarks import expected_landmark_vertices, expected_landmarks, pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def _graph(n, edges, name, seed=3):
    g = P.csr_from_edges(n, np.asarray(edges, np.int64), name)
    return g, P.degree_rank(g, "random", seed)


def path(n):
    return _graph(n, np.stack([np.arange(n - 1), np.arange(1, n)], 1), f"path{n}")


def hubs(*degrees):
    """A path of 700 vertices with stars of the given degrees along it, and
    a second component of a path of 40."""
    e = [(i, i + 1) for i in range(699)] + [(700 + i, 701 + i) for i in range(39)]
    at = 740
    for j, d in enumerate(degrees):
        c = 50 + 90 * j
        e += [(c, at + i) for i in range(d - 2)]
        at += d - 2
    return _graph(at, e, "hubs")


GRAPHS = {
    "path8": lambda: path(8),
    "path9": lambda: path(9),
    "path31": lambda: path(31),
    "path32": lambda: path(32),
    "path33": lambda: path(33),
    "path640": lambda: path(640),
    "hubs": lambda: hubs(63, 64, 65, 1500),
    "grid21x33": lambda: _graph(21 * 33, [(v, v + s) for v in range(21 * 33) for s in (1, 33)
                                          if (s == 33 and v + 33 < 21 * 33) or (s == 1 and v % 33 != 32)], "grid"),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("k", [1, 32, 65, 128])
def test_searches_equal_bfs(pspc, name, k):  # noqa: F811
    g, rank = GRAPHS[name]()
    ix = pspc.Index.from_graph(g, rank, landmarks=k)
    try:
        ids = expected_landmark_vertices(g, rank, k)
        assert ix.landmark_vertices().tolist() == ids
        assert np.array_equal(ix.landmarks(), expected_landmarks(g, rank, k, ids))
    finally:
        ix.free()
