"""Dense graphs: few candidates in very many messages.  Receivers with more than
65,536 messages (neighbours' new labels) are gathered by a block."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1906_12018_gb300 import graphs as G
from paper_1906_12018_gb300 import plb

from gpu_util import assert_labels_equal, to_device

pytestmark = pytest.mark.gpu


def complete(n):
    i, j = np.triu_indices(n, 1)
    return G.clean_csr(n, np.concatenate([i, j]).astype(np.int32), np.concatenate([j, i]).astype(np.int32))


def in_block_tier(n):
    """Receivers of round 2 of K_n in rank order: neighbour a sends a hubs, so v's
    neighbours send n (n - 1) / 2 - v in all."""
    return int(np.sum(n * (n - 1) // 2 - np.arange(1, n) > 65536))


@pytest.mark.parametrize("n", [362, 363, 364, 370, 513, 600])
def test_complete_graphs(n):
    g = complete(n)
    order = np.arange(n, dtype=np.int32)
    ref = O.pll(g.off, g.col, order)
    rp, col, o = to_device(g, order)
    lab = plb.build(rp, col, o)
    assert_labels_equal(lab, ref)
    if n < 513:  # (longer label rows go to the block tier for their length)
        assert lab.stats()["tier_vertices"][1] == in_block_tier(n)
    wt = torch.ones(col.numel(), dtype=torch.uint8, device="cuda")
    assert_labels_equal(plb.build_weighted(rp, col, wt, o), ref)
    for side in plb.build_directed(rp, col, o):
        assert_labels_equal(side, ref)


@pytest.mark.parametrize("opts", [{}, {"use_graph": 1}], ids=["host", "graph"])
def test_dense_random_graphs_in_a_union(opts):
    """Graphs around the largest whose messages stay below the limit (362
    vertices: those need no top-hub columns), with sparse ones between."""
    rng = np.random.default_rng(8)
    gs = []
    for n, p in ((361, 0.95), (40, 0.1), (363, 0.97), (420, 0.9), (5, 0.5), (362, 1.0), (500, 0.8)):
        s, t = np.nonzero(np.triu(rng.random((n, n)) < p, 1))
        gs.append(G.clean_csr(n, np.concatenate([s, t]).astype(np.int32), np.concatenate([t, s]).astype(np.int32)))
    orders = [rng.permutation(g.n).astype(np.int32) for g in gs]
    sets = plb.build_batch([to_device(g, o) for g, o in zip(gs, orders)], plb.default_options(**opts))
    for i, (g, o) in enumerate(zip(gs, orders)):
        assert_labels_equal(sets[i], O.pll(g.off, g.col, o), f"part {i}")
    assert sets[0].stats()["tier_vertices"][1] > 0
