"""Direct-address merging of candidates (vertices with many pulled
entries): every entry of the index equals the definition or the oracle on
graphs that reach the edges of its windows, tables and count bound."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import pspc_inputs as P
from tests import _graphs as G
from tests.test_gpu_parity import _check_whole_index, assert_index_equal, gpu_index

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pspc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2212_00977_gb300 as lib

    lib.load()
    return lib


WINDOWS = [
    (15, 8, "degree", {}),                    # three windows of ids
    (14, 16, "random", {}),                   # hubs anywhere: long rows over several windows, no table of window starts
    (14, 16, "degree", {"granular": True}),   # only the heaviest vertices
    (14, 8, "degree", {"landmarks": -1}),     # every candidate goes to the label scans
    (13, 16, "degree", {"max_ctas": 3}),      # a few CTAs take every vertex
]


@pytest.mark.parametrize("scale,ef,order,kw", WINDOWS)
def test_windows_and_rows(pspc, scale, ef, order, kw):
    """With distance balls, whose rows stand for the member bitmaps and for
    rule 2, at level 3."""
    g = P.rmat(scale, ef, *P.RMAT_ABCD, seed=5)
    rank = P.degree_rank(g, "id") if order == "degree" else G.random_rank(g.n, 4)
    ix = gpu_index(pspc, g, rank, **kw)
    level = ix.level_stats()[2]
    assert level["unique_candidates"] == level["entries"]
    _check_whole_index(g, rank, *ix.export())
    ix.free()


@pytest.mark.parametrize("scale,ef,order,kw", WINDOWS)
def test_windows_and_rows_without_balls(pspc, scale, ef, order, kw):
    """The same graphs among isolated vertices, too many for balls: member
    bitmaps, the marking walk of level 3 (in two rounds of ids where the
    graph's are spread over all of them), the filter and the scans."""
    g = P.rmat(scale, ef, *P.RMAT_ABCD, seed=5)
    n = 170_000 if order == "random" else 131_100
    g = P.csr_from_edges(n, g.edges(), "among isolated")
    rank = P.degree_rank(g, "id") if order == "degree" else G.random_rank(g.n, 4)
    ix = gpu_index(pspc, g, rank, **kw)
    for level in ix.level_stats()[2:4]:
        assert level["unique_candidates"] > level["entries"] and level["raw_candidates"] > 1 << 19
    _check_whole_index(g, rank, *ix.export())
    ix.free()


@pytest.mark.parametrize("m", [255, 256, 257])
def test_fewest_pulled_entries(pspc, m):
    """Vertices that pull 510, 512 and 514 entries: either side of the line
    between the hash and the windows."""
    g = G.hub_ladder(m, 6)
    rank = np.arange(g.n, dtype=np.int32)
    ref = oracle.OracleIndex(g, rank).export()
    for kw in ({}, {"landmarks": -1}, {"max_ctas": 1}):
        ix = gpu_index(pspc, g, rank, **kw)
        assert_index_equal(ix, ref)
        ix.free()


@pytest.mark.parametrize("m,depth", [(1500, 34), (1300, 66)])
def test_counts_up_to_the_bound(pspc, m, depth):
    """Ladder vertices pull 2m entries with counts 2^(level - 1): sums are
    merged in 32 bits while the bound allows, in 64 bits beyond it, through
    2^32 and 2^64."""
    g = G.hub_ladder(m, depth)
    rank = np.arange(g.n, dtype=np.int32)
    ref = oracle.OracleIndex(g, rank).export()
    ix = gpu_index(pspc, g, rank)
    assert_index_equal(ix, ref)
    ix.free()


def test_batch_of_dense_graphs(pspc):
    """Graphs of a batch at id ranges that start inside a window's width."""
    graphs = [P.rmat(s, 16, *P.RMAT_ABCD, seed=s) for s in (12, 11, 13)]
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
