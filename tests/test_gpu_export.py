"""pspc_export gathered on the device, in chunks of 4 Mi entries: the same
bytes as the form ordered on the host, which a failing allocation (the first,
second or third of a call) leads to; one chunk and several, words and plain
hubs, vertices with no arcs."""
from __future__ import annotations

import numpy as np
import pytest

import pspc_inputs as P
from tests.test_gpu_landmarks import pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def _edges(n, e, name):
    g = P.csr_from_edges(n, np.asarray(e, np.int64).reshape(-1, 2), name)
    return g, P.degree_rank(g, "random", 3)


def _grid(w, h):
    v = np.arange(w * h).reshape(h, w)
    return np.concatenate([np.stack([v[:, :-1].ravel(), v[:, 1:].ravel()], 1),
                           np.stack([v[:-1].ravel(), v[1:].ravel()], 1)])


GRAPHS = {
    "one": lambda: _edges(1, [], "one"),
    "isolated": lambda: _edges(70, [(3, 5), (5, 9)], "isolated"),
    "ba2000": lambda: P.workload("ba2000")[:2],
    "grid40": lambda: _edges(1600, _grid(40, 40), "grid40"),
    "grid100": lambda: _edges(10000, _grid(100, 100), "grid100"),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_device_and_host_forms_agree(pspc, name):  # noqa: F811
    g, rank = GRAPHS[name]()
    ix = pspc.Index.from_graph(g, rank)
    try:
        got = ix.export()
        if name == "grid100":
            assert len(got[1]) > 2 * (4 << 20)  # three chunks
        for failing in (0, 1, 2):
            pspc.inject_alloc_failure(failing)
            try:
                ref = ix.export()
            finally:
                pspc.inject_alloc_failure(-1)
            for a, b in zip(got, ref):
                assert a.dtype == b.dtype and np.array_equal(a, b)
    finally:
        ix.free()


@pytest.mark.parametrize("name", ["isolated", "grid100"])
def test_other_errors_are_reported(pspc, name):  # noqa: F811
    """The host form is for a device without room, not for a CUDA error."""
    g, rank = GRAPHS[name]()
    ix = pspc.Index.from_graph(g, rank)
    try:
        for failing in range(3 if name == "grid100" else 2):  # the scan allocates beyond 4,096 vertices
            pspc.inject_alloc_failure(failing, pspc.PSPC_E_CUDA)
            try:
                with pytest.raises(pspc.PSPCError) as e:
                    ix.export()
            finally:
                pspc.inject_alloc_failure(-1)
            assert e.value.code == pspc.PSPC_E_CUDA
        assert len(ix.export()[1]) == ix.stats()["entries"]
    finally:
        ix.free()
