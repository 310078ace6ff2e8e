"""Performance cases of the labeling library: what a program that uses it has it do.

Each case is one call (or one user-level step) through the public entry points
of ``paper_1906_12018_gb300.plb``: label a graph, label a batch of graphs,
label a directed or a weighted graph, answer distance queries, order the
vertices.  The graphs are seeded random power-law graphs, generated on the
GPU; the seed changes every edge, weight and pair.  Label sets differ in size
from seed to seed, so the caller's buffers are sized for the case and the
unused tail stays zero.
"""
import math

import numpy as np
import torch

from paper_1906_12018_gb300 import graphs
from paper_1906_12018_gb300 import plb

RMAT = (0.57, 0.19, 0.19)  # the generator's quadrant probabilities a, b, c (d = 0.05)


def listed():
    return [
        # the smallest graph that is labeled in earnest: launches, host reads and allocations count
        {"name": "build_rmat_4k", "op": "build", "graph": "rmat", "n": 1 << 12, "degree": 16, "gamma": 0.0},
        # one graph of the labeling service's job stream; an odd size, with isolated vertices
        {"name": "build_chunglu_61k", "op": "build", "graph": "chunglu", "n": 61007, "degree": 10, "gamma": 2.3},
        # a whole social-network-like graph of a million vertices
        {"name": "build_chunglu_1m", "op": "build", "graph": "chunglu", "n": 1 << 20, "degree": 16, "gamma": 2.1},
        # the largest graph of the benchmark: 4.2M ids, 64M edges, about 1.8G labels
        {"name": "build_rmat_4m", "op": "build", "graph": "rmat", "n": 1 << 22, "degree": 32, "gamma": 0.0},
        # many small graphs of uneven sizes (1K-64K vertices, half R-MAT, half Chung-Lu) in one call
        {"name": "batch_200", "op": "batch", "graphs": 200, "first": 0},
        # a directed graph: both label sets
        {"name": "directed_rmat_1m", "op": "directed", "graph": "rmat", "n": 1 << 20, "degree": 16, "gamma": 0.0},
        # a weighted graph, weights 1..7
        {"name": "weighted_chunglu_1m", "op": "weighted", "graph": "chunglu", "n": 1 << 20, "degree": 16,
         "gamma": 2.1, "max_weight": 7},
        # the largest query request of the serving loop on the largest label set (long rows)
        {"name": "query_rmat_4m", "op": "query", "graph": "rmat", "n": 1 << 22, "degree": 32, "gamma": 0.0,
         "pairs": 65536},
        # a small request on a label set of short rows: a launch
        {"name": "query_chunglu_1m_small", "op": "query", "graph": "chunglu", "n": 1 << 20, "degree": 16,
         "gamma": 2.1, "pairs": 997},
        # requests on many resident label sets, coalesced into one launch
        {"name": "query_multi", "op": "multi", "graphs": 32, "first": 300, "n": 1 << 20, "degree": 16, "gamma": 2.1,
         "pairs": 1000003},
        # d(s -> t) from the two label sets of a directed graph
        {"name": "query_directed", "op": "query_directed", "graph": "rmat", "n": 1 << 18, "degree": 16, "gamma": 0.0,
         "pairs": 65536},
        # the vertex order that every labeling starts from
        {"name": "order_4m", "op": "order", "graph": "chunglu", "n": 4000037, "degree": 16, "gamma": 2.1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, lo, hi, max_degree):
    n = _log_int(rng, lo, hi)
    if rng.random() < 0.5:
        return {"graph": "rmat", "n": n, "degree": rng.randint(6, max_degree), "gamma": 0.0}
    return {"graph": "chunglu", "n": n, "degree": rng.randint(4, max_degree), "gamma": round(rng.uniform(2.05, 2.6), 3)}


def draw(rng):
    op = rng.choice(["build", "build", "build", "batch", "directed", "weighted", "query", "query", "multi",
                     "query_directed", "order"])
    if op == "build":
        return {"op": op, **_draw_graph(rng, 1 << 10, 3 << 19, 24)}
    if op == "batch":
        return {"op": op, "graphs": _log_int(rng, 5, 300), "first": rng.randrange(1600)}
    if op == "directed":
        return {"op": op, **_draw_graph(rng, 1 << 10, 3 << 18, 16)}
    if op == "weighted":
        return {"op": op, **_draw_graph(rng, 1 << 10, 3 << 18, 16), "max_weight": rng.choice([1, 3, 7, 7, 7, 12])}
    if op == "query":
        return {"op": op, **_draw_graph(rng, 1 << 10, 1 << 20, 24), "pairs": _log_int(rng, 1, 1 << 18)}
    if op == "multi":
        return {"op": op, "graphs": _log_int(rng, 2, 200), "first": rng.randrange(1600),
                "n": _log_int(rng, 1 << 10, 1 << 20), "degree": 16, "gamma": 2.1, "pairs": _log_int(rng, 100, 1 << 20)}
    if op == "query_directed":
        return {"op": op, **_draw_graph(rng, 1 << 10, 1 << 18, 16), "pairs": _log_int(rng, 1, 1 << 18)}
    return {"op": op, "graph": "chunglu", "n": _log_int(rng, 1 << 10, 4 << 20), "degree": rng.randint(2, 20),
            "gamma": 2.1}


# ------------------------------------------------------------------ inputs
def _rmat_arcs(n, m, gen):
    """m R-MAT arcs over the ids [0, n) (arcs with an id >= n are drawn again)."""
    a, b, c = RMAT
    levels = max(1, (n - 1).bit_length())
    src, dst, have = [], [], 0
    while have < m:
        k = m if (1 << levels) == n else int(1.6 * (m - have)) + 64
        s = torch.zeros(k, dtype=torch.int64, device="cuda")
        t = torch.zeros(k, dtype=torch.int64, device="cuda")
        for _ in range(levels):
            u = torch.rand(k, generator=gen, device="cuda")
            s.mul_(2).add_(u >= a + b)
            t.mul_(2).add_(((u >= a) & (u < a + b)) | (u >= a + b + c))
        if (1 << levels) != n:
            keep = (s < n) & (t < n)
            s, t = s[keep], t[keep]
        src.append(s[: m - have])
        dst.append(t[: m - have])
        have += src[-1].numel()
    return torch.cat(src), torch.cat(dst)


def _chung_lu_arcs(n, m, gamma, gen):
    """m arcs, both ends drawn with probability proportional to (i + 1)^(-1 / (gamma - 1))."""
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda").pow_(-1.0 / (gamma - 1.0))
    cdf = torch.cumsum(w, 0)
    u = torch.rand(2 * m, generator=gen, device="cuda", dtype=torch.float64).mul_(cdf[-1])
    e = torch.searchsorted(cdf, u).clamp_(max=n - 1)
    return e[:m], e[m:]


def _rows(n, key):
    """CSR (int64 offsets, int32 columns) of the sorted unique keys src * n + dst."""
    bounds = torch.arange(n + 1, dtype=torch.int64, device="cuda") * n
    return torch.searchsorted(key, bounds), (key % n).to(torch.int32)


def _arcs(case, gen):
    n, m = case["n"], max(1, case["degree"] * case["n"] // 2)
    if case["op"] in ("directed", "query_directed"):
        m = case["degree"] * n
    s, t = _rmat_arcs(n, m, gen) if case["graph"] == "rmat" else _chung_lu_arcs(n, m, case["gamma"], gen)
    keep = s != t
    return n, s[keep], t[keep]


def _undirected(case, gen):
    """Symmetric CSR without self-loops and duplicates; R-MAT graphs without their isolated ids."""
    n, s, t = _arcs(case, gen)
    key = torch.unique(torch.cat((s * n + t, t * n + s)))
    row_ptr, col = _rows(n, key)
    if case["graph"] == "rmat":
        used = row_ptr[1:] > row_ptr[:-1]
        col = (torch.cumsum(used, 0) - 1).to(torch.int32)[col.long()]
        row_ptr = torch.cat((row_ptr[:1], row_ptr[1:][used]))
    return row_ptr.contiguous(), col.contiguous()


def _directed(case, gen):
    """Out-arcs as a CSR and the in + out degree order (descending, ties by id)."""
    n, s, t = _arcs(case, gen)
    key = torch.unique(s * n + t)
    row_ptr, col = _rows(n, key)
    deg = (row_ptr[1:] - row_ptr[:-1]) + torch.bincount(col.long(), minlength=n)
    order = torch.sort(deg, descending=True, stable=True).indices.to(torch.int32)
    return row_ptr, col.contiguous(), order


def _weights(row_ptr, col, top, seed):
    """One uniform weight in [1, top] per edge: both of its arcs hash to the same value."""
    n = row_ptr.numel() - 1
    u = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr[1:] - row_ptr[:-1])
    v = col.long()
    x = torch.minimum(u, v) * 0x9E3779B1 + torch.maximum(u, v) * 0x85EBCA6B + seed * 0x27D4EB2F
    for _ in range(2):
        x = (x ^ (x >> 29)) * 0x2545F4914F6CDD1D
    return (1 + ((x >> 33) & 0x3FFFFFFF) % top).to(torch.uint8)


def _small_case(i):
    n = graphs.small_graph_size(i)
    if i % 2 == 0:
        return {"op": "build", "graph": "rmat", "n": n, "degree": 16, "gamma": 0.0}
    return {"op": "build", "graph": "chunglu", "n": n, "degree": 10, "gamma": 2.3}


def _label_model(case):
    """Labels of one label set, roughly (a power law in n and m / n)."""
    n, per = case["n"], max(case["degree"], 2) / 2.0
    if case["op"] in ("directed", "query_directed"):
        per = float(case["degree"])
    return n * math.exp(-0.7 + 0.305 * math.log(n) + 0.756 * math.log(per))


def _label_buffers(rows, labels):
    """Caller-owned label arrays for up to `labels` entries, and some more."""
    cap = int(2.0 * labels) + 64 * rows // 8 + 4096
    return {"off": torch.zeros(rows, dtype=torch.int64, device="cuda"),
            "hub": torch.zeros(cap, dtype=torch.int32, device="cuda"),
            "dist": torch.zeros(cap, dtype=torch.uint8, device="cuda")}


def _pairs(n, q, gen):
    return torch.randint(0, n, (q, 2), generator=gen, device="cuda", dtype=torch.int32)


def prepare(case, seed):
    op = case["op"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    state = {"op": op}
    if op in ("build", "weighted", "query"):
        row_ptr, col = _undirected(case, gen)
        order = plb.degree_order(row_ptr)
        if op == "query":
            state["labels"] = plb.build(row_ptr, col, order)
            state["pairs"] = _pairs(row_ptr.numel() - 1, case["pairs"], gen)
            return state
        state["graph"] = (row_ptr, col, order)
        state["out"] = _label_buffers(case["n"] + 1, _label_model(case))
        if op == "weighted":
            state["weight"] = _weights(row_ptr, col, case["max_weight"], int(seed))
    elif op in ("directed", "query_directed"):
        state["graph"] = _directed(case, gen)
        if op == "directed":
            state["out"] = [_label_buffers(case["n"] + 1, _label_model(case)) for _ in range(2)]
        else:
            state["labels"] = plb.build_directed(*state.pop("graph"))
            state["pairs"] = _pairs(case["n"], case["pairs"], gen)
    elif op == "batch":
        small = [_small_case(case["first"] + i) for i in range(case["graphs"])]
        state["graphs"] = []
        for c in small:
            row_ptr, col = _undirected(c, gen)
            state["graphs"].append((row_ptr, col, plb.degree_order(row_ptr)))
        state["out"] = _label_buffers(sum(c["n"] + 1 for c in small), sum(_label_model(c) for c in small))
    elif op == "multi":
        cases = [_small_case(case["first"] + i) for i in range(case["graphs"])]
        sets = []
        for c in cases:
            row_ptr, col = _undirected(c, gen)
            sets.append((row_ptr, col, plb.degree_order(row_ptr)))
        big = {"op": "build", "graph": "chunglu", "n": case["n"], "degree": case["degree"], "gamma": case["gamma"]}
        row_ptr, col = _undirected(big, gen)
        state["labels"] = plb.build_batch(sets) + [plb.build(row_ptr, col, plb.degree_order(row_ptr))]
        # a third of the pairs on the large set, the others spread over the small ones
        q, m = case["pairs"], len(state["labels"])
        which = torch.randint(0, m - 1, (q,), generator=gen, device="cuda", dtype=torch.int32)
        large = torch.rand(q, generator=gen, device="cuda") < 1.0 / 3.0
        which[large] = m - 1
        sizes = torch.tensor([s.n for s in state["labels"]], device="cuda")[which.long()]
        u = torch.rand((q, 2), generator=gen, device="cuda", dtype=torch.float64)
        state["pairs"] = (u * sizes[:, None]).to(torch.int32)
        state["which"] = which
    else:  # order
        state["row_ptr"], _ = _undirected(case, gen)
    return state


# --------------------------------------------------------------------- run
def _take(labels, out):
    """The label arrays in the caller's own tensors; the set goes back to the library."""
    off, hub, dist = labels.device_arrays()
    out["off"][: off.numel()].copy_(off)
    out["hub"][: hub.numel()].copy_(hub)
    out["dist"][: dist.numel()].copy_(dist)
    labels.free()
    return {"off": out["off"], "hub": out["hub"], "dist": out["dist"], "max_dist": labels.max_dist}


def run(state):
    op = state["op"]
    if op == "build":
        return _take(plb.build(*state["graph"]), state["out"])
    if op == "weighted":
        row_ptr, col, order = state["graph"]
        return _take(plb.build_weighted(row_ptr, col, state["weight"], order), state["out"])
    if op == "directed":
        l_in, l_out = plb.build_directed(*state["graph"])
        return {"in": _take(l_in, state["out"][0]), "out": _take(l_out, state["out"][1])}
    if op == "batch":
        sets = plb.build_batch(state["graphs"])
        parts = [s.device_arrays() for s in sets]
        out = state["out"]
        for k, name in enumerate(("off", "hub", "dist")):
            torch.cat([p[k] for p in parts], out=out[name][: sum(p[k].numel() for p in parts)])
        del parts
        for s in sets:
            s.free()
        return {"off": out["off"], "hub": out["hub"], "dist": out["dist"]}
    if op == "query":
        return state["labels"].query(state["pairs"])
    if op == "query_directed":
        l_in, l_out = state["labels"]
        return plb.query_directed(l_out, l_in, state["pairs"])
    if op == "multi":
        return plb.query_multi(state["labels"], state["which"], state["pairs"])
    return plb.degree_order(state["row_ptr"])


# -------------------------------------------------------------------- work
def _build_bytes(case):
    """CSR and order read once; offsets, hubs and distances written once."""
    n = case["n"]
    arcs = case["degree"] * n * (1 if case["op"] != "weighted" else 1.25)
    sets = 2 if case["op"] == "directed" else 1
    return 8.0 * (n + 1) + 4.0 * arcs + 4.0 * n + sets * (8.0 * (n + 1) + 5.0 * _label_model(case))


def work(case):
    op = case["op"]
    if op in ("build", "directed", "weighted"):
        b = _build_bytes(case)
    elif op == "batch":
        b = sum(_build_bytes(_small_case(case["first"] + i)) for i in range(case["graphs"]))
    elif op == "order":
        b = 8.0 * (case["n"] + 1) + 4.0 * case["n"]
    else:
        # per pair: the pair, its answer and the two label rows
        if op == "multi":
            small = [_small_case(case["first"] + i) for i in range(case["graphs"])]
            rows = sum(_label_model(c) / c["n"] for c in small) / len(small) * 2.0 / 3.0
            rows += _label_model({**case, "graph": "chunglu"}) / case["n"] / 3.0
        else:
            rows = _label_model(case) / case["n"]
        b = case["pairs"] * (12.0 + (4.0 if op == "multi" else 0.0) + 2 * 5.0 * rows)
    return {"bytes": b, "flops": 0.0}


# ------------------------------------------------------------------- exact
def _exact_labels(row_ptr, col, order):
    """Def. of the canonical labels from all-pairs distances (small graphs): in
    rank order, h is a hub of v unless a hub of both that outranks h already
    gives d(h, v)."""
    n = row_ptr.numel() - 1
    rank = torch.empty(n, dtype=torch.int64, device="cuda")
    rank[order.long()] = torch.arange(n, device="cuda")
    adj = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr[1:] - row_ptr[:-1])
    adj[rank[src], rank[col.long()]] = 1.0
    far = 1e6
    dist = torch.full((n, n), far, dtype=torch.float64, device="cuda")
    reach = torch.eye(n, dtype=torch.float64, device="cuda")
    dist[reach > 0] = 0.0
    d, more = 0, True
    while more:
        d += 1
        nxt = (reach @ adj) > 0
        new = nxt & (dist >= far)
        dist[new] = float(d)
        more = bool(new.any())
        reach = new.to(torch.float64)
    lab = torch.full((n, n), far, dtype=torch.float64, device="cuda")  # [hub, vertex]
    for h in range(n):
        best = (lab[:h, h, None] + lab[:h]).amin(0) if h else torch.full((n,), far, device="cuda")
        ok = (dist[h] < far) & (dist[h] < best)
        ok[:h] = False
        lab[h, ok] = dist[h, ok]
    by_id = lab.t()[rank]  # rows by id, columns hubs in rank order
    has = by_id < far
    off = torch.cat((torch.zeros(1, dtype=torch.int64, device="cuda"), torch.cumsum(has.sum(1), 0)))
    return off, has.nonzero()[:, 1].to(torch.int32), by_id[has].to(torch.uint8)


def exact(case, seed):
    op = case["op"]
    if op == "order":
        row_ptr = prepare(case, seed)["row_ptr"].cpu().numpy()
        deg = np.diff(row_ptr)
        order = np.lexsort((np.arange(deg.size), -deg)).astype(np.int32)
        return order
    if op == "build" and case["n"] <= 4096:
        state = prepare(case, seed)
        off, hub, dist = _exact_labels(*state["graph"])
        out = state["out"]
        out["off"][: off.numel()] = off
        out["hub"][: hub.numel()] = hub
        out["dist"][: dist.numel()] = dist
        return {"off": out["off"], "hub": out["hub"], "dist": out["dist"], "max_dist": int(dist.max())}
    return None
