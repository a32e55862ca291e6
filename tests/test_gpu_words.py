"""Queries on packed words (hub, distance and small count in 32 bits): every
way of running them (a warp per few pairs, sorted and unsorted, a CTA per
pair, look-ups of short labels, runs of one source) equals breadth-first path
counting, with counts that fit a word, that do not, and that overflow."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import pspc_inputs as P
from tests import _graphs as G
from tests.test_gpu_parity import gpu_index, gpu_query, pspc  # noqa: F401

pytestmark = pytest.mark.gpu


def _layers(width: int, depth: int):
    """depth layers of width vertices, consecutive ones completely joined:
    width^(k-1) shortest paths over k layers."""
    e = [(a * width + i, (a + 1) * width + j) for a in range(depth - 1) for i in range(width) for j in range(width)]
    return P.csr_from_edges(width * depth, np.array(e), f"layers{width}x{depth}")


def _async(ix, pairs):
    import torch

    q = len(pairs)
    p = torch.from_numpy(pairs).cuda()
    d = torch.empty(q, dtype=torch.uint16, device="cuda")
    c = torch.empty(q, dtype=torch.uint64, device="cuda")
    f = torch.empty(q, dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    ix.query_async(p, d, c, f, err)
    torch.cuda.synchronize()
    assert int(err[0]) == 0
    return d.cpu().numpy(), c.cpu().numpy(), f.cpu().numpy()


@pytest.mark.parametrize("make,seed", [
    (lambda: (P.workload("rmat16_ef2")[0], "degree"), 1),  # ids fill a word's hub bits; isolated vertices
    (lambda: (G.bipartite_2m(1600), "id"), 2),             # labels of several hash segments, all tied
    (lambda: (_layers(24, 16), "random"), 3),              # counts from 1 to beyond 2^64 in 16 levels
    (lambda: (G.hub_ladder(500, 14), "id"), 4),            # counts around what a word holds
])
def test_words_equal_path_counting(pspc, make, seed):  # noqa: F811
    g, order = make()
    rank = {"degree": lambda: P.degree_rank(g, "id"), "id": lambda: np.arange(g.n, dtype=np.int32),
            "random": lambda: G.random_rank(g.n, seed)}[order]()
    rng = np.random.default_rng(seed)
    last = np.argsort(rank)[-3:]  # the lowest-ranked vertices
    src = rng.integers(0, g.n, 60)
    pairs = np.concatenate([np.stack([np.repeat(src, 300), rng.integers(0, g.n, 18000)], 1),
                            np.stack([np.repeat(last, 500), rng.integers(0, g.n, 1500)], 1),
                            np.stack([rng.integers(0, g.n, 1500), np.repeat(last, 500)], 1)]).astype(np.int32)
    pairs = pairs[rng.permutation(len(pairs))]
    rd, rc, rf, _ = oracle.spc_pairs(g, pairs)
    ix = gpu_index(pspc, g, rank)
    if seed == 3:
        assert ix.stats()["levels"] == 16 and rf.any() and not rf.all()
    for group in (0, 256, pspc.PSPC_QUERY_BY_SOURCE, pspc.PSPC_QUERY_BY_SOURCE_HASH, 16):
        ix.set_query_group(group)
        for d, c, f in (gpu_query(ix, pairs), _async(ix, pairs)):
            assert np.array_equal(d, rd) and np.array_equal(c, rc) and np.array_equal(f, rf), group
        for k in (1, 33, 1000):  # few pairs: a CTA each where labels are long
            d, c, f = _async(ix, pairs[:k])
            assert np.array_equal(d, rd[:k]) and np.array_equal(c, rc[:k]) and np.array_equal(f, rf[:k]), (group, k)
    ix.free()
