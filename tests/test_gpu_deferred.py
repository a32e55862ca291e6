"""Deep levels' label scans, queued and run by later launches: the index
equals the oracle's with so few landmarks that most candidates are undecided
and many are pruned by their scans (segments closed with entries taken out),
with more undecided candidates than the queue holds, for the warp-per-vertex
and the CTA-per-vertex kernels, and with few CTAs."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import pspc_inputs as P
from tests import _graphs as G
from tests.test_gpu_parity import _check_whole_index, assert_index_equal, gpu_index, pspc  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,order", [("grid90", "degree"), ("grid70", "random")])
def test_deferred_scans(pspc, name, order):  # noqa: F811
    g, rank, _ = P.workload(name)
    if order == "random":
        rank = G.random_rank(g.n, 9)
    ref = oracle.OracleIndex(g, rank).export()
    for kw in (dict(landmarks=1), dict(landmarks=1, warp_levels=-1), dict(landmarks=40, max_ctas=2), dict(granular=True),
               dict(landmarks=3, arena_entries=1)):
        ix = gpu_index(pspc, g, rank, **kw)
        assert_index_equal(ix, ref)
        ls = ix.level_stats()
        assert sum(l["entries"] for l in ls) + g.n == len(ref.hub)
        ix.free()


@pytest.mark.parametrize("kw", [{}, {"warp_levels": -1}])
def test_more_scans_than_the_queue_holds(pspc, kw):  # noqa: F811
    g, rank, _ = P.workload("grid100")
    ix = gpu_index(pspc, g, rank, landmarks=1, **kw)
    undecided = [l["unique_candidates"] - l["landmark_pruned"] - l["landmark_proven"] for l in ix.level_stats()]
    assert max(undecided) > max(4 * g.n, 1 << 16)
    _check_whole_index(g, rank, *ix.export())
    ix.free()


def test_odd_cycles(pspc):  # noqa: F811
    """Not bipartite: witnesses at both distance sums d-1 and d-2."""
    rng = np.random.default_rng(3)
    base = G.grid(64)
    extra = np.array([(v, v + 65) for v in rng.integers(0, 62 * 64, 700) if v % 64 < 63])
    g = P.csr_from_edges(base.n, np.concatenate([base.edges(), extra]), "diagonals")
    rank = P.degree_rank(g, "random", 5)
    ref = oracle.OracleIndex(g, rank).export()
    for kw in (dict(), dict(landmarks=2), dict(landmarks=2, warp_levels=-1)):
        ix = gpu_index(pspc, g, rank, **kw)
        assert_index_equal(ix, ref)
        ix.free()


@pytest.mark.parametrize("n,m", [(2500, 3), (4001, 4)])
def test_shallow_levels_that_defer(pspc, n, m):  # noqa: F811
    """Levels 4 to 15 with 2^18 pulled entries, 2,048 active vertices or more
    and no distance ball (which a chosen label map rules out)."""
    g = P.barabasi_albert(n, m, 7)
    rank = P.degree_rank(g, "random", 5)
    ref = oracle.OracleIndex(g, rank).export()
    for kw in (dict(map_kind=1), dict(map_kind=2, landmarks=1), dict(map_kind=3, landmarks=2, warp_levels=15),
               dict(map_kind=1, granular=True)):
        ix = gpu_index(pspc, g, rank, **kw)
        assert any(l["raw_candidates"] >= 1 << 18 and l["active_vertices"] >= 2048 for l in ix.level_stats()[3:])
        assert_index_equal(ix, ref)
        ix.free()
