"""The cost pass of graphs of small degrees (up to 32: four lanes walk a
vertex's arcs) and the general one equal the oracle at the line between
them, with rows of every remainder, isolated vertices, dense prefixes, the
push paradigm, a retried arena and batches."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import pspc_inputs as P
from tests import _graphs as G
from tests.test_gpu_parity import assert_index_equal, gpu_index, pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def bounded(n, most, seed):
    """A random graph whose largest degree is `most`, with a chain so that
    it is deep, and a few isolated vertices at the end."""
    rng = np.random.default_rng(seed)
    deg = np.zeros(n, int)
    edges = {(v, v + 1) for v in range(n - 9)}
    for a, b in edges:
        deg[a] += 1
        deg[b] += 1
    for _ in range(n // 2):
        a = int(rng.integers(0, n - 40))
        b = a + int(rng.integers(2, 40))
        if b < n - 8 and (a, b) not in edges and deg[a] < most and deg[b] < most:
            edges.add((a, b))
            deg[a] += 1
            deg[b] += 1
    hub = n // 3
    for v in range(n - 8):
        if deg[hub] >= most:
            break
        e = (min(hub, v), max(hub, v))
        if v != hub and e not in edges and deg[v] < most:
            edges.add(e)
            deg[hub] += 1
            deg[v] += 1
    assert deg.max() == most
    return P.csr_from_edges(n, np.array(sorted(edges)), f"most{most}")


@pytest.mark.parametrize("most", [4, 31, 32, 33])
@pytest.mark.parametrize("n", [127, 128, 129, 700])
def test_levels_equal_the_oracle(pspc, n, most):  # noqa: F811
    g = bounded(n, most, n + most)
    rank = P.degree_rank(g, "random", 5)
    ref = oracle.OracleIndex(g, rank).export()
    for kw in (dict(), dict(paradigm=1), dict(arena_entries=1), dict(landmarks=-1, granular=True)):
        ix = gpu_index(pspc, g, rank, **kw)
        assert_index_equal(ix, ref)
        ix.free()


def test_batch_of_small_degrees(pspc):  # noqa: F811
    graphs = [(g, P.degree_rank(g, "random", 2)) for g in (G.grid(9), G.path(50), G.cycle(33), bounded(90, 32, 1))]
    with pspc.Index.build_batch([(g.n, g.row_ptr, g.col, r) for g, r in graphs]) as ix:
        base = 0
        for g, r in graphs:
            ref = oracle.OracleIndex(g, r).export()
            off, hub, dist, cnt, ovf = ix.export_vertices(np.arange(base, base + g.n, dtype=np.int32))
            assert np.array_equal(off, ref.off) and np.array_equal(hub - base, ref.hub)
            assert np.array_equal(dist, ref.dist) and np.array_equal(cnt, ref.cnt)
            base += g.n
