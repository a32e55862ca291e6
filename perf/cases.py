"""Performance cases of the SPC hub-label library.

A case is one pass of a user's program through the package's public calls
(``Index.build``, ``Index.build_batch``, ``Index.query``,
``Index.query_async``, ``Index.export``) on seeded synthetic graphs of the
families the repository is used on: power-law R-MAT and Barabasi-Albert
graphs (social and web graphs) and rectangular grids with a tenth of their
edges deleted (road networks). ``do`` says which pass:

* ``build``: build the index, use it once (answer ``q`` pairs, or copy the
  whole index to the host when ``q`` is 0), free it.
* ``batch``: the same for a batch of graphs in one build, its pairs
  answered by one stream-ordered call.
* ``query``: answer ``q`` pairs on a resident index, from device or host
  buffers; ``async`` takes the stream-ordered call into kept buffers.

Graphs and pairs are made on the GPU from the seed alone. Every output is a
whole number (distance, count modulo 2^64, overflow flag), so every
tolerance is exact.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2212_00977_gb300 as pspc

RMAT_ABCD = (0.57, 0.19, 0.19, 0.05)
GRID_DELETED = 0.10


# --------------------------------------------------------------- the cases

def listed():
    return [
        # The smallest build: a small social graph handed over as host
        # arrays and the finished index saved (exported) by the program.
        # Launches, host round trips and the export's gather count here.
        {"name": "build_ba_2k_export", "do": "build", "graph": "ba", "n": 2000, "m": 4, "q": 0, "host": True},
        # A build request of the serving loop (granular CTAs, host arrays),
        # followed by one request's worth of pairs.
        {"name": "build_ba_20k_granular", "do": "build", "graph": "ba", "n": 20011, "m": 5, "q": 4096, "host": True,
         "granular": True},
        # The ordinary single-graph build: R-MAT of 65,536 vertices, edge
        # factor 16, then as many pairs as vertices.
        {"name": "build_rmat_64k", "do": "build", "graph": "rmat", "n": 65536, "ef": 16, "q": 65536},
        # The large build: R-MAT of 2^20 vertices, edge factor 8, then 10^7
        # pairs (the power-law half of the benchmark).
        {"name": "build_rmat_1m", "do": "build", "graph": "rmat", "n": 1 << 20, "ef": 8, "q": 10_000_000},
        # A small road network: many levels with little work in each.
        {"name": "build_grid_61x67", "do": "build", "graph": "grid", "w": 61, "h": 67, "q": 20_000},
        # The large road network of the benchmark, then 10^7 pairs.
        {"name": "build_grid_256x256", "do": "build", "graph": "grid", "w": 256, "h": 256, "q": 10_000_000},
        # Many small graphs built at once, every one queried by one
        # stream-ordered call.
        {"name": "batch_ba_96", "do": "batch", "graphs": 96, "n_lo": 500, "n_hi": 20000, "q": 960_000},
        # One pair at a time: the latency of the smallest call.
        {"name": "query_one", "do": "query", "graph": "rmat", "n": 1 << 18, "ef": 8, "q": 1, "how": "device"},
        # A batch of the serving loop: a few requests' pairs on a resident
        # index, stream-ordered.
        {"name": "query_async_1500", "do": "query", "graph": "rmat", "n": 1 << 18, "ef": 8, "q": 1500, "how": "async"},
        # 10^6 pairs on the ordinary graph.
        {"name": "query_rmat_64k_1m", "do": "query", "graph": "rmat", "n": 65536, "ef": 16, "q": 1_000_000,
         "how": "device"},
        # Many pairs per source on a road network (long labels).
        {"name": "query_grid_128x128_2m", "do": "query", "graph": "grid", "w": 128, "h": 128, "q": 2_000_000,
         "how": "device"},
        # Pairs and answers in host memory.
        {"name": "query_host_rmat_256k_200k", "do": "query", "graph": "rmat", "n": 1 << 18, "ef": 8, "q": 200_003,
         "how": "host"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, rmat_top, grid_top):
    kind = rng.choice(["rmat", "rmat", "grid", "ba"])
    if kind == "rmat":
        n = _log_int(rng, 1000, rmat_top)
        return {"graph": "rmat", "n": n, "ef": rng.randint(4, max(4, min(16, (1 << 22) // n)))}
    if kind == "ba":
        return {"graph": "ba", "n": _log_int(rng, 500, 100_000), "m": rng.randint(2, 8)}
    area = math.exp(rng.uniform(math.log(400), math.log(grid_top)))
    w = max(8, int(math.sqrt(area * rng.uniform(0.5, 1.0))))
    return {"graph": "grid", "w": w, "h": max(8, int(area / w))}


def draw(rng):
    do = rng.choice(["build", "build", "build", "batch", "query", "query", "query"])
    if do == "batch":
        lo = _log_int(rng, 100, 2000)
        k = _log_int(rng, 3, 96)
        return {"do": "batch", "graphs": k, "n_lo": lo, "n_hi": lo * rng.randint(2, 8), "q": k * _log_int(rng, 100, 10_000)}
    if do == "build":
        case = {"do": "build", **_draw_graph(rng, 400_000, 30_000), "host": rng.random() < 0.3,
                "granular": rng.random() < 0.2, "reduce_shell": rng.random() < 0.15}
        n = _vertices(case)
        case["q"] = 0 if n < 5000 and not case["reduce_shell"] and rng.random() < 0.4 else _log_int(rng, 1, 400_000)
        return case
    case = {"do": "query", **_draw_graph(rng, 300_000, 16_000), "how": rng.choice(["device", "device", "async", "host"])}
    case["q"] = _log_int(rng, 1, 3_000_000 if case["how"] == "device" else 300_000)
    return case


# ------------------------------------------------------------- the graphs

def _csr(n, src, dst):
    """Symmetric CSR (rows ascending) of an undirected edge list, without
    self-loops and duplicates: (row_ptr int64, col int32) on the GPU."""
    keep = src != dst
    src, dst = src[keep], dst[keep]
    key = torch.unique(torch.cat([src * n + dst, dst * n + src]))
    row = torch.div(key, n, rounding_mode="floor")
    rp = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    rp[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return rp, (key - row * n).to(torch.int32)


def _rank(rp, gen):
    """Degree-descending order, ties at random, as a rank array."""
    n = rp.numel() - 1
    tie = torch.randperm(n, generator=gen, device=rp.device)
    order = torch.argsort((rp[1:] - rp[:-1]) * (-n) + tie)
    rank = torch.empty(n, dtype=torch.int32, device=rp.device)
    rank[order] = torch.arange(n, dtype=torch.int32, device=rp.device)
    return rank


def _rmat(n, ef, gen):
    """ef * n R-MAT samples over the next power of two; those outside
    [0, n) are dropped."""
    a, b, c, _ = RMAT_ABCD
    count = ef * n
    src = torch.zeros(count, dtype=torch.int64, device="cuda")
    dst = torch.zeros(count, dtype=torch.int64, device="cuda")
    for bit in range(max(1, (n - 1).bit_length())):
        r = torch.rand(count, generator=gen, device="cuda")
        src |= (r >= a + b).to(torch.int64) << bit
        dst |= (((r >= a) & (r < a + b)) | (r >= a + b + c)).to(torch.int64) << bit
    keep = (src < n) & (dst < n)
    return _csr(n, src[keep], dst[keep])


def _grid(w, h, gen):
    """w x h 4-neighbour grid with a tenth of its edges deleted."""
    ids = torch.arange(w * h, dtype=torch.int64, device="cuda").reshape(h, w)
    src = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
    dst = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
    keep = torch.randperm(src.numel(), generator=gen, device="cuda")[int(GRID_DELETED * src.numel()):]
    return _csr(w * h, src[keep], dst[keep])


def _ba(n, m, gen):
    """Preferential attachment, all edges at once: edge i leaves vertex
    m + i // m for the end found at a uniformly drawn earlier end of an
    edge (an odd end is another edge's target: followed to its source)."""
    edges = torch.arange(m * max(1, n - m), dtype=torch.int64, device="cuda")
    source = m + torch.div(edges, m, rounding_mode="floor")
    first = m * torch.div(edges, m, rounding_mode="floor")  # edges of earlier vertices
    pick = (torch.rand(edges.numel(), generator=gen, device="cuda", dtype=torch.float64) * (2 * first)).to(torch.int64)
    at = torch.div(pick, 2, rounding_mode="floor")
    jump = torch.where((pick % 2 == 1) & (edges >= m), at, edges)  # the edge whose target it takes
    target = torch.where(edges < m, edges, source[at])             # known unless it takes another's
    for _ in range(max(1, edges.numel()).bit_length()):
        jump = jump[jump]
    return _csr(n, source, target[jump])


def _renamed(rp, col, rank, gen):
    """The same graph and order under other vertex ids."""
    n = rp.numel() - 1
    new = torch.randperm(n, generator=gen, device="cuda")
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    rp, col = _csr(n, new[src], new[col.long()])
    moved = torch.empty_like(rank)
    moved[new] = rank
    return rp, col, moved


def _graph(case, gen):
    """(n, row_ptr, col, rank) on the GPU. Where the whole index is copied
    out, the seed only names the vertices, so that it always has one size."""
    kind = case["graph"]
    whole = case["do"] == "build" and case["q"] == 0
    made = torch.Generator(device="cuda").manual_seed(1) if whole else gen
    if kind == "rmat":
        rp, col = _rmat(case["n"], case["ef"], made)
    elif kind == "grid":
        rp, col = _grid(case["w"], case["h"], made)
    else:
        rp, col = _ba(case["n"], case["m"], made)
    rank = _rank(rp, made)
    if whole:
        rp, col, rank = _renamed(rp, col, rank, gen)
    return rp.numel() - 1, rp, col, rank


def _pairs(n, q, gen):
    return torch.randint(0, n, (q, 2), generator=gen, device="cuda", dtype=torch.int32)


# --------------------------------------------------------------- one pass

def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    do, q = case["do"], int(case["q"])
    if do == "batch":
        span = max(1, case["n_hi"] - case["n_lo"])
        size = (case["n_lo"] + torch.randint(0, span + 1, (case["graphs"],), generator=gen, device="cuda")).tolist()
        ms = torch.randint(2, 9, (case["graphs"],), generator=gen, device="cuda").tolist()
        graphs, base, pairs = [], 0, []
        for n, m in zip(size, ms):
            rp, col = _ba(n, m, gen)
            graphs.append((n, rp, col, _rank(rp, gen)))
            pairs.append(_pairs(n, q // case["graphs"], gen) + base)
            base += n
        pairs = torch.cat(pairs)
        return {"case": case, "graphs": graphs, "pairs": pairs, **_buffers(len(pairs))}
    n, rp, col, rank = _graph(case, gen)
    pairs = _pairs(n, q, gen) if q else None
    if do == "build":
        if case.get("host"):
            rp, col, rank = rp.cpu().numpy(), col.cpu().numpy(), rank.cpu().numpy()
            pairs = None if pairs is None else pairs.cpu().numpy()
        return {"case": case, "n": n, "graph": (rp, col, rank), "pairs": pairs}
    index = pspc.Index.build(n, rp, col, rank)
    if case["how"] == "host":
        return {"case": case, "index": index, "pairs": pairs.cpu().numpy()}
    if case["how"] == "async":
        return {"case": case, "index": index, "pairs": pairs, **_buffers(q)}
    return {"case": case, "index": index, "pairs": pairs}


def _buffers(q):
    """Answer buffers that a program with stream-ordered calls keeps."""
    return {"dist": torch.empty(q, dtype=torch.uint16, device="cuda"),
            "count": torch.empty(q, dtype=torch.uint64, device="cuda"),
            "overflow": torch.empty(q, dtype=torch.uint8, device="cuda"),
            "err": torch.zeros(1, dtype=torch.int32, device="cuda")}


def _signed(dist, count, overflow):
    """The same answers seen as signed numbers of the same width (not every
    tensor operation takes the unsigned types)."""
    if isinstance(dist, np.ndarray):
        return {"dist": dist.view(np.int16), "count": count.view(np.int64), "overflow": overflow}
    return {"dist": dist.view(torch.int16), "count": count.view(torch.int64), "overflow": overflow}


def run(state):
    case = state["case"]
    if case["do"] == "query":
        index = state["index"]
        if case["how"] == "async":
            index.query_async(state["pairs"], state["dist"], state["count"], state["overflow"], state["err"])
            return {**_signed(state["dist"], state["count"], state["overflow"]), "err": state["err"]}
        return _signed(*index.query(state["pairs"]))
    if case["do"] == "batch":
        with pspc.Index.build_batch(state["graphs"]) as index:
            index.query_async(state["pairs"], state["dist"], state["count"], state["overflow"], state["err"])
            s = index.stats()
        return {**_signed(state["dist"], state["count"], state["overflow"]), "err": state["err"],
                "entries": s["entries"], "levels": s["levels"]}
    opts = {k: bool(case[k]) for k in ("granular", "reduce_shell") if case.get(k)}
    with pspc.Index.build(state["n"], *state["graph"], **opts) as index:
        s = index.stats()
        size = {"entries": s["entries"], "levels": s["levels"], "overflow_entries": s["overflow_entries"]}
        if state["pairs"] is None:
            off, hub, dist, cnt, ovf = index.export()
            return {**size, "off": off, "hub": hub, **_signed(dist, cnt, ovf)}
        return {**size, **_signed(*index.query(state["pairs"]))}


# ------------------------------------------------------------- what it takes

def _vertices(case):
    return case["w"] * case["h"] if case["graph"] == "grid" else case["n"]


def _arcs(case):
    """Directed arcs, about: self-loops and duplicates of R-MAT dropped."""
    if case["graph"] == "grid":
        return 4 * (1 - GRID_DELETED) * case["w"] * case["h"]
    return 1.7 * case["ef"] * case["n"] if case["graph"] == "rmat" else 2 * case["m"] * case["n"]


def _entries(case):
    """Label entries of the index, about: fits to measured index sizes."""
    n = _vertices(case)
    if case["graph"] == "grid":
        return 0.19 * n ** 1.94
    if case["graph"] == "rmat":
        return 0.64 * n ** 1.59 * (case["ef"] / 8) ** 0.68
    return 0.87 * n ** 1.62 * (case["m"] / 4) ** 1.2


def _query_work(q, n, entries):
    """The pairs and their answers, and each label that they touch once
    (hub and distance, 6 bytes an entry); one comparison for each entry of
    a pair's two labels."""
    touched = 1 - math.exp(-2 * q / n)
    return {"bytes": q * (8 + 11) + touched * 6 * entries, "flops": q * 2 * entries / n}


def work(case):
    if case["do"] == "batch":
        n = (case["n_lo"] + case["n_hi"]) / 2
        one = {"graph": "ba", "n": n, "m": 5}
        parts = [(case["graphs"], one, case["q"] / case["graphs"])]
    else:
        parts = [(1, case, case["q"])]
    total = {"bytes": 0.0, "flops": 0.0}
    for k, g, q in parts:
        n, e = _vertices(g), _entries(g)
        w = _query_work(q, n, e) if q else {"bytes": 14.0 * e, "flops": 0.0}
        total["bytes"] += k * w["bytes"]
        total["flops"] += k * w["flops"]
        if case["do"] != "query":  # the graph and its order read, the index written
            total["bytes"] += k * (12 * n + 4 * _arcs(g) + 14 * e)
            total["flops"] += k * e
    return total


def tolerance(case):
    return "exact"


# ------------------------------------------------- the definition, in int64

def _neighbour_sums(rp, col, x):
    """out[v] = sum of x[w] over the neighbours w of v, rows of an int64
    matrix, modulo 2^64."""
    src = torch.repeat_interleave(torch.arange(rp.numel() - 1, device=rp.device), rp[1:] - rp[:-1])
    return torch.zeros_like(x).index_add_(0, src, x[col.long()])


def _paths(rp, col, sources, allowed):
    """Distances (-1: unreached) and numbers of shortest paths modulo 2^64
    from each source (a column), through vertices with allowed[v, column]."""
    n, k = rp.numel() - 1, sources.numel()
    dist = torch.full((n, k), -1, dtype=torch.int64, device=rp.device)
    count = torch.zeros((n, k), dtype=torch.int64, device=rp.device)
    col_id = torch.arange(k, device=rp.device)
    dist[sources, col_id] = 0
    count[sources, col_id] = 1
    front, d = count.clone(), 0
    reach = (front != 0).to(torch.int64)
    while bool(reach.any()):
        d += 1
        new = (_neighbour_sums(rp, col, reach) > 0) & (dist < 0) & allowed
        front = torch.where(new, _neighbour_sums(rp, col, front), torch.zeros_like(front))
        dist = torch.where(new, torch.full_like(dist, d), dist)
        count = torch.where(new, front, count)
        reach = new.to(torch.int64)
    return dist, count


def exact(case, seed):
    """Plain breadth-first counting, where it is quick: the answers of a
    query call with few pairs, and the whole index of a small graph (hub w
    is in the label of v when the paths through vertices ranked below w are
    as short as any). Overflow flags are left out: 64 bits do not show
    them."""
    if case["do"] == "batch" or case.get("reduce_shell"):
        return None
    state_case = {**case, "host": False}
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n, rp, col, rank = _graph(state_case, gen)
    arcs = int(rp[-1])
    if case["q"] == 0:
        if n > 4500 or case["graph"] == "grid":
            return None
        rank = rank.long()
        order = torch.argsort(rank)
        below = rank[:, None] >= torch.arange(n, device="cuda")[None, :]
        dist, _ = _paths(rp, col, order, torch.ones_like(below))
        part, count = _paths(rp, col, order, below)
        label = (part >= 0) & (part == dist)
        v, w = torch.nonzero(label, as_tuple=True)  # by vertex, then by hub rank
        off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        off[1:] = torch.cumsum(label.sum(1), 0)
        return {"entries": int(label.sum()), "levels": int(part[label].max()) + 1, "overflow_entries": None,
                "off": off, "hub": order[w].to(torch.int32), "dist": part[label].to(torch.int16),
                "count": count[label], "overflow": None}
    pairs = _pairs(n, case["q"], gen).long()
    if case["q"] > 64 or arcs * case["q"] > 1 << 31 or (case["graph"] == "grid" and n > 5000):
        return None
    dist, count = _paths(rp, col, pairs[:, 0], torch.ones((n, case["q"]), dtype=torch.bool, device="cuda"))
    at = torch.arange(case["q"], device="cuda")
    answer = {"dist": dist[pairs[:, 1], at].to(torch.int16), "count": count[pairs[:, 1], at], "overflow": None}
    if case["do"] == "query":
        return {**answer, "err": None} if case["how"] == "async" else answer
    return {**answer, "entries": None, "levels": None, "overflow_entries": None}
