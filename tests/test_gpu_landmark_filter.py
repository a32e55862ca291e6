"""The landmark filter's row widths: every landmark count that fills a row
of 16-byte words differently (4 or 8 lanes to a row, whole and part words),
on a deep grid and on a graph in several pieces, where a landmark is
undefined for whole components; the index equals the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import pspc_inputs as P
from tests import _graphs as G
from tests.test_gpu_parity import assert_index_equal, gpu_index, pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def _pieces():
    """A 20 x 20 grid, a 12 x 12 grid, a long path and isolated vertices."""
    a, b, c = G.grid(20), G.grid(12), G.path(60)
    e = np.concatenate([a.edges(), b.edges() + a.n, c.edges() + a.n + b.n])
    return P.csr_from_edges(a.n + b.n + c.n + 3, e, "pieces")


@pytest.mark.parametrize("k", [1, 7, 8, 9, 31, 32, 33, 65, 100, 128])
def test_every_row_width(pspc, k):  # noqa: F811
    for g, rank in ((P.workload("grid32")[:2]), (_pieces(), None)):
        rank = G.random_rank(g.n, 7) if rank is None else rank
        ref = oracle.OracleIndex(g, rank).export()
        for kw in ({}, {"warp_levels": -1}, {"warp_levels": 1000}):
            ix = gpu_index(pspc, g, rank, landmarks=k, **kw)
            assert_index_equal(ix, ref)
            ix.free()
