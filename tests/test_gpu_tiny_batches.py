"""Batches of very many very small graphs: a graph whose receivers cannot reach
the block tier takes no top-hub columns."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1906_12018_gb300 import graphs as G
from paper_1906_12018_gb300 import plb

from gpu_util import assert_labels_equal, to_device

pytestmark = pytest.mark.gpu


def small(n, seed):
    rng = np.random.default_rng(seed)
    g = G.from_edges(n, [(int(a), int(b)) for a, b in rng.integers(0, n, (2 * n, 2)) if a != b] or [(0, 1)])
    return g, G.degree_order(g)


def test_memory_of_many_tiny_graphs():
    """4,096 graphs of 16 vertices need little more than the labels, masks, tables
    and rows that the same vertices need as one graph: per graph a descriptor,
    its offsets, 16 x 24 bytes of union rows and fewer than 64 arcs (below 1 KB
    in all; 4 KB allow for the allocator's rounding).  A quad of columns each
    would take 28,672 bytes."""
    k, n = 4096, 16
    parts = [small(n, s) for s in range(8)]
    dev = [to_device(g, o) for g, o in parts]
    row_ptr = np.concatenate([[0]] + [np.cumsum(np.diff(parts[i % 8][0].off)) for i in range(k)])
    ends = np.concatenate([[0], np.cumsum([parts[i % 8][0].nnz for i in range(k)])])
    off = np.concatenate([parts[i % 8][0].off[:-1] + ends[i] for i in range(k)] + [ends[-1:]])
    assert off.size == k * n + 1 and row_ptr.size == off.size
    col = np.concatenate([parts[i % 8][0].col + n * i for i in range(k)])
    order = np.concatenate([parts[i % 8][1] + n * i for i in range(k)])
    one = [torch.from_numpy(np.ascontiguousarray(a, dtype=t)).cuda()
           for a, t in ((off, np.int64), (col, np.int32), (order, np.int32))]

    def peak(fn):
        torch.cuda.synchronize()
        before = plb.memory_stats(reset=True)
        sets = fn()
        torch.cuda.synchronize()
        high = plb.memory_stats()["used_high"] - before["used"]
        return high, sets

    base, lab = peak(lambda: [plb.build(*one)])
    total = lab[0].total
    lab[0].free()
    many, sets = peak(lambda: plb.build_batch([dev[i % 8] for i in range(k)]))
    assert sum(s.total for s in sets) == total
    for i in (0, 7, k - 1):
        g, o = parts[i % 8]
        assert_labels_equal(sets[i], O.pll(g.off, g.col, o), f"part {i}")
    for s in sets:
        s.free()
    assert many - base <= k * 4096, (many, base)


@pytest.mark.parametrize("opts,least", [({}, 512), ({"warp_label_cap": 40}, 40), ({"warp_cand_cap": 32}, 32),
                                        ({"use_graph": 1}, 512)], ids=["default", "label", "candidates", "graph"])
def test_graphs_around_the_size_without_columns(opts, least):
    """Unions of graphs with and without columns, dense enough that the larger
    ones fill the block tier where the options allow it."""
    rng = np.random.default_rng(5)
    gs = []
    for n in (least - 1, 3, least, least + 1, 1, 2 * least, least + 2):
        s, t = np.nonzero(np.triu(rng.random((n, n)) < min(0.9, 14.0 / n), 1))
        gs.append(G.clean_csr(n, np.concatenate([s, t]).astype(np.int32), np.concatenate([t, s]).astype(np.int32)))
    orders = [rng.permutation(g.n).astype(np.int32) for g in gs]
    sets = plb.build_batch([to_device(g, o) for g, o in zip(gs, orders)], plb.default_options(**opts))
    for i, (g, o) in enumerate(zip(gs, orders)):
        assert_labels_equal(sets[i], O.pll(g.off, g.col, o), f"part {i}")
        rp, col, od = to_device(g, o)
        assert_labels_equal(plb.build(rp, col, od, **opts), O.pll(g.off, g.col, o), f"alone {i}")
