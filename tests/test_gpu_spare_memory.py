"""Memory that only makes a build faster (distance balls, direct-address
slabs, the queue of scans): a build for which there is no room goes on
without it, or with less of it, gives it back when the index needs more
room, and its index is the same. One allocation after another fails, alone
or with those after it."""
from __future__ import annotations

import numpy as np
import pytest

import pspc_inputs as P
from tests.test_gpu_parity import pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def _balls_used(ls):
    """Levels that prune by a ball count nothing but their survivors."""
    return sum(0 < l["unique_candidates"] == l["entries"] and l["landmark_pruned"] == l["landmark_proven"] == 0
               for l in ls[2:])


def _rmat():
    g = P.rmat(13, 16, *P.RMAT_ABCD, seed=2)
    return g, P.degree_rank(g, "id")


def _batch(lib, **kw):
    graphs = [P.barabasi_albert(n, m, n) for n, m in ((3000, 5), (129, 4), (2000, 8))]
    return lib.Index.build_batch([(g.n, g.row_ptr, g.col, P.degree_rank(g, "id")) for g in graphs], **kw)


BUILDS = {
    # balls and slabs; the same with an arena that grows beside them; balls of a batch; the queue
    "rmat": (lambda lib, **kw: lib.Index.from_graph(*_rmat(), **kw), {}, 5),
    "small arena": (lambda lib, **kw: lib.Index.from_graph(*_rmat(), **kw), dict(arena_entries=1), 7),
    "batch": (_batch, {}, 6),
    "grid": (lambda lib, **kw: lib.Index.from_graph(*P.workload("grid90")[:2], **kw), dict(landmarks=8), 3),
}


# 13 failures: the slabs of 1,216 CTAs halved down to one CTA's, which then
# takes the place of the balls
@pytest.mark.parametrize("name,count", [(name, 1) for name in BUILDS] + [("rmat", 13)])
def test_allocations_fail(pspc, name, count):  # noqa: F811
    make, kw, least = BUILDS[name]
    with make(pspc, **kw) as ix:
        ref, balls = ix.export(), 0 if name == "grid" else _balls_used(ix.level_stats())
    assert balls > 0 or name == "grid"
    went_on = without_balls = k = 0
    reported = True
    while reported:  # allocation k fails, until there is no such allocation
        pspc.inject_alloc_failure(k, pspc.PSPC_E_CUDA, count=1)
        try:
            make(pspc, **kw).free()
            reported = False
        except pspc.PSPCError as e:  # only a lack of room is worked around
            assert e.code == pspc.PSPC_E_CUDA, k
        pspc.inject_alloc_failure(k, count=count)
        try:
            ix = make(pspc, **kw)
        except pspc.PSPCError as e:
            assert reported and e.code == pspc.PSPC_E_NOMEM, k
        else:
            with ix:
                for a, b in zip(ix.export(), ref):
                    assert np.array_equal(a, b), k
                went_on += reported
                without_balls += reported and _balls_used(ix.level_stats()) < balls
        finally:
            pspc.inject_alloc_failure(-1)
        k += 1
        assert k < 400
    assert k > 25 and went_on >= (least if count == 1 else 1)
    assert without_balls >= (0 if name == "grid" else 4 if count == 1 else 1)
