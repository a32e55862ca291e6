"""Label scans whose filter is nearly full: the two labels meet at one hub
only, among thousands of entries that match the filter by chance, so the
matches are looked up several times within a row of entries. The index
equals the oracle's where the scans run in a warp of their own, split over
a CTA's warps, and queued."""
from __future__ import annotations

import numpy as np
import pytest

import pspc_inputs as P
from tests import _graphs as G
from tests.test_gpu_parity import _check_whole_index, gpu_index, pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def crowded_cycles(cycles: int, near: int, far: int, crowd: int, group: int = 100, short: bool = True, more=None):
    """Even cycles through one vertex h, and an order in which each vertex u
    across h has to drop the candidate (h, d), d = near + far + 2, for one
    hub x alone: x lies on the shorter way, `near` from u and `far` (at least
    2) from h. A hundred more hubs are that near to u (half of them ranked
    above x, half below) and `crowd` more that far from h, none of them in
    both labels: a vertex on top of the order joins them. It joins the x too
    (short), or u pulls the crowd's entries from x's side at level d. more: a
    graph put beside, ranked below. Returns (graph, rank, h, the u)."""
    edges, tops, ahead, xs, behind, middle, low = [], [], [], [], [], [], []
    n = 0

    def new(k, group_of):
        nonlocal n
        ids = list(range(n, n + k))
        n += k
        group_of.extend(ids)
        return ids

    def chain(a, b, length):  # a path of `length` edges through new low vertices
        at = [a] + (new(length - 1, low) + [b] if b is not None else new(length, low))
        edges.extend(zip(at[:-1], at[1:]))
        return at[-1]

    top = new(1, tops)[0]
    crowded = new(crowd, tops)
    h = new(1, middle)[0]
    trunk = chain(h, None, far - 2)
    for i in range(0, crowd, group):
        m = chain(trunk, None, 1)
        edges.extend((m, a) for a in crowded[i:i + group])
    edges.extend((top, a) for a in crowded)
    us = []
    for _ in range(cycles):
        u = new(1, low)[0]
        us.append(u)
        x = new(1, xs)[0]
        if short:
            edges.append((top, x))
        chain(u, x, near)
        chain(x, h, far)
        chain(u, h, near + far + 2)
        trunk = chain(u, None, near - 1)
        for b in new(50, ahead) + new(50, behind):
            edges.extend([(trunk, b), (top, b)])
    if more is not None:
        edges.extend((n + a, n + b) for a, b in more.edges())
        new(more.n, low)
    rank = np.empty(n, np.int32)
    rank[tops + ahead + xs + behind + middle + low] = np.arange(n, dtype=np.int32)
    return P.csr_from_edges(n, np.array(edges), "crowdedcycles"), rank, h, us


CASES = {
    # near, far, crowd...: the filter's 8,192 bits are all set (32,768 where the scans are queued)
    "warp": (dict(cycles=12, near=1, far=2, crowd=12000), dict(map_kind=3, warp_levels=1000)),
    "warp, no landmarks": (dict(cycles=12, near=1, far=2, crowd=12000),
                           dict(map_kind=3, warp_levels=1000, landmarks=-1)),
    "split over four warps": (dict(cycles=12, near=5, far=10, crowd=12000),
                              dict(map_kind=3, warp_levels=-1, landmarks=1)),
    # more than 131,072 vertices: no distance ball
    "split over eight warps": (dict(cycles=4, near=2, far=2, crowd=12000, short=False,
                                    more=P.csr_from_edges(131072, np.zeros((0, 2), np.int64))), {}),
    # 2,048 active vertices and 2^18 pulled entries: queued
    "queued": (dict(cycles=12, near=1, far=2, crowd=40000, group=400, more=G.grid(64)),
               dict(map_kind=3, warp_levels=1000)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_one_witness_among_chance_matches(pspc, name):  # noqa: F811
    make, kw = CASES[name]
    g, rank, h, us = crowded_cycles(**make)
    ix = gpu_index(pspc, g, rank, **kw)
    if name == "queued":
        level = ix.level_stats()[make["near"] + make["far"] + 1]  # of distance d
        assert level["raw_candidates"] >= 1 << 18 and level["active_vertices"] >= 2048
    off, hub, dist, cnt, ovf = ix.export()
    for u in us:
        assert h not in hub[off[u]:off[u + 1]]
    _check_whole_index(g, rank, off, hub, dist, cnt, ovf)
    ix.free()
