"""Levels that prune by distance balls: every entry of the index equals the
oracle's or the definition's on graphs whose levels use them from level 3 or
only in between; rows longer than a warp's slice; batches of graphs of
very different sizes; balls caught up over several levels."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import pspc_inputs as P
from tests import _graphs as G
from tests.test_gpu_parity import _check_whole_index, assert_index_equal, gpu_index, pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def _star_of_paths(arms: int, length: int, hubs: int):
    """Hubs joined to the first vertex of every arm: rows of `arms` arcs and
    distances up to 2 * length."""
    e = [(h, hubs + a * length) for h in range(hubs) for a in range(arms)]
    e += [(hubs + a * length + i, hubs + a * length + i + 1) for a in range(arms) for i in range(length - 1)]
    return P.csr_from_edges(hubs + arms * length, np.array(e), "starpaths")


@pytest.mark.parametrize("make", [
    lambda: (P.barabasi_albert(6000, 6, 3), "degree"),
    lambda: (P.barabasi_albert(4097, 3, 5), "random"),
    lambda: (P.rmat(13, 12, *P.RMAT_ABCD, seed=2), "degree"),
    lambda: (_star_of_paths(700, 5, 300), "random"),  # rows of 700 and 301 arcs, ten levels
])
def test_single_graphs(pspc, make):  # noqa: F811
    g, order = make()
    rank = P.degree_rank(g, "id") if order == "degree" else G.random_rank(g.n, 6)
    for kw in ({}, {"landmarks": -1}, {"granular": True}):
        ix = gpu_index(pspc, g, rank, **kw)
        _check_whole_index(g, rank, *ix.export())
        ix.free()


def _sparse(n, seed):
    e = np.random.default_rng(seed).integers(0, n, (3 * n // 2, 2))
    return P.csr_from_edges(n, e[e[:, 0] != e[:, 1]], "sparse")


@pytest.mark.parametrize("batch", [False, True])
def test_balls_caught_up(pspc, batch):  # noqa: F811
    """Sparse random graphs, whose candidates are few at first: the first
    level with a ball brings it four steps or more at once, and the last
    levels go without."""
    graphs = [_sparse(n, 3) for n in ((4000, 2500) if batch else (4000,))]
    ranks = [G.random_rank(g.n, 6) for g in graphs]
    if batch:
        ix = pspc.Index.build_batch([(g.n, g.row_ptr, g.col, r) for g, r in zip(graphs, ranks)])
    else:
        ix = gpu_index(pspc, graphs[0], ranks[0])
    by_ball = [l["unique_candidates"] == l["entries"] > 1 << 15 and l["landmark_pruned"] == 0 for l in ix.level_stats()]
    assert not any(by_ball[2:5]) and any(by_ball[5:8]) and not any(by_ball[-3:])
    base = 0
    for g, r in zip(graphs, ranks):
        off, hub, dist, cnt, ovf = ix.export_vertices(np.arange(base, base + g.n, dtype=np.int32))
        _check_whole_index(g, r, off, hub - base, dist, cnt, ovf)
        base += g.n
    ix.free()


def test_batch_of_uneven_graphs(pspc):  # noqa: F811
    graphs = [P.barabasi_albert(n, m, n) for n, m in ((3001, 5), (40, 3), (5000, 7), (129, 4), (128, 2), (2000, 8))]
    graphs.insert(3, P.csr_from_edges(1, np.zeros((0, 2), np.int64)))
    ranks = [P.degree_rank(g, "id") for g in graphs]
    ix = pspc.Index.build_batch([(g.n, g.row_ptr, g.col, r) for g, r in zip(graphs, ranks)])
    base = 0
    for g, r in zip(graphs, ranks):
        ref = oracle.OracleIndex(g, r).export()
        off, hub, dist, cnt, ovf = ix.export_vertices(np.arange(base, base + g.n, dtype=np.int32))
        assert np.array_equal(off, ref.off) and np.array_equal(hub - base, ref.hub)
        assert np.array_equal(dist, ref.dist) and np.array_equal(cnt, ref.cnt) and np.array_equal(ovf, ref.ovf)
        base += g.n
    ix.free()
