"""Distances at which nothing is accepted: weighted rounds without a label at
their distance, and directed builds whose two sides need different numbers of
rounds.  The labels known at such a distance are those of the distance below it,
and a witness among them still refutes a candidate (bit-exact against the oracle)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1906_12018_gb300 import graphs as G
from paper_1906_12018_gb300 import plb

from gpu_util import assert_labels_equal, to_device

pytestmark = pytest.mark.gpu

FORCED = dict(warp_cand_cap=32, warp_label_cap=16, block_cand_cap=64, block_label_cap=24, block_threads=64)

# leaves of the receiver and options that take it to the block tier: by its label
# row (lowered and default options), and as a receiver with more than 2,048 arcs
RECEIVERS = [pytest.param(20, FORCED, id="lowered"), pytest.param(520, {}, id="default"),
             pytest.param(2100, {}, id="split")]


def weighted_csr(n, edges):
    """Symmetric CSR and arc weights of (u, v, weight) edges (no duplicates)."""
    u, v, w = (np.array(x) for x in zip(*edges))
    g = G.clean_csr(n, u.astype(np.int32), v.astype(np.int32))
    key = {(min(a, b), max(a, b)): x for a, b, x in zip(u.tolist(), v.tolist(), w.tolist())}
    src = np.repeat(np.arange(n), np.diff(g.off)).tolist()
    return g, np.array([key[(min(a, b), max(a, b))] for a, b in zip(src, g.col.tolist())], dtype=np.uint8)


def check_weighted(g, wt, order, **opts):
    rp, col, o = to_device(g, order)
    lab = plb.build_weighted(rp, col, torch.from_numpy(wt).cuda(), o, **opts)
    assert_labels_equal(lab, O.pll_weighted(g.off, g.col, wt, order))
    return lab


@pytest.mark.parametrize("leaves,opts", RECEIVERS)
def test_weighted_witness_below_an_empty_distance(leaves, opts):
    """0 is joined to 1 and to the last vertex by weight 2, these two by weight 5:
    candidate 1 at distance 5 has the witness 0 (2 + 2), and no label has
    distance 3 = 5 - 2."""
    v = leaves + 2
    edges = [(0, 1, 2), (0, v, 2), (1, v, 5)] + [(i, v, 2) for i in range(2, v)]
    g, wt = weighted_csr(v + 1, edges)
    lab = check_weighted(g, wt, np.arange(v + 1, dtype=np.int32), **opts)
    assert lab.stats()["tier_vertices"][1] > 0


@pytest.mark.parametrize("weights", [(2, 5), (3, 4), (3, 7), (2, 7), (2, 3, 7), (4, 6)], ids=str)
@pytest.mark.parametrize("seed", range(6))
def test_weighted_random_graphs_with_empty_distances(weights, seed):
    rng = np.random.default_rng(100 * weights[0] + 10 * weights[-1] + seed)
    n = int(rng.integers(60, 160))
    s, t = np.nonzero(np.triu(rng.random((n, n)) < 6.0 / n, 1))
    g, wt = weighted_csr(n, list(zip(s.tolist(), t.tolist(), rng.choice(weights, len(s)).tolist())))
    for order in (G.degree_order(g), rng.permutation(n).astype(np.int32)):
        check_weighted(g, wt, order, **FORCED)


def check_directed(g, order, **opts):
    ref_in, ref_out = O.pll_directed(g.off, g.col, g.off_in, g.col_in, order)
    lin, lout = plb.build_directed(torch.from_numpy(g.off).cuda(), torch.from_numpy(g.col).cuda(),
                                   torch.from_numpy(order).cuda(), **opts)
    assert_labels_equal(lin, ref_in, "in")
    assert_labels_equal(lout, ref_out, "out")
    return lin, lout


@pytest.mark.parametrize("leaves,opts", RECEIVERS)
@pytest.mark.parametrize("flip", [False, True], ids=["in ends first", "out ends first"])
def test_directed_witness_on_a_side_that_has_finished(leaves, opts, flip):
    """v -> 0 -> 1 and v -> a -> b -> 1: candidate 1 at distance 3 of v has the
    witness 0 (1 + 1); nothing is reached over two arcs on the other side, which
    accepts nothing after round 1."""
    a, b, v = leaves + 2, leaves + 3, leaves + 4
    arcs = [(v, 0), (0, 1), (v, a), (a, b), (b, 1)] + [(v, i) for i in range(2, a)]
    src, dst = (np.array(x, dtype=np.int32) for x in zip(*arcs))
    if flip:
        src, dst = dst, src
    lin, lout = check_directed(G.directed_csr(v + 1, src, dst), np.arange(v + 1, dtype=np.int32), **opts)
    rounds = (lin.stats()["rounds"], lout.stats()["rounds"])
    assert rounds[flip] < rounds[not flip]
    assert (lin if flip else lout).stats()["tier_vertices"][1] > 0


@pytest.mark.parametrize("seed", range(8))
def test_directed_random_graphs(seed):
    rng = np.random.default_rng(seed)
    for _ in range(25):
        n = int(rng.integers(70, 140))
        m = int(n * rng.uniform(1.5, 4))
        g = G.directed_csr(n, rng.integers(0, n, m), rng.integers(0, n, m))
        check_directed(g, G.directed_degree_order(g), **FORCED)
        check_directed(g, rng.permutation(n).astype(np.int32), **FORCED)
