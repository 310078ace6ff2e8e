"""The gather + prune tiers at the edges of their tables and masks, against the
oracle (bit-exact)."""
import numpy as np
import pytest

import oracle as O
from paper_1906_12018_gb300 import graphs as G
from paper_1906_12018_gb300 import plb

from gpu_util import assert_labels_equal, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [{}, {"use_graph": 1}, {"batch_hubs": 300},
                                  {"warp_cand_cap": 32, "warp_label_cap": 16, "block_cand_cap": 64,
                                   "block_label_cap": 24, "block_threads": 64}],
                         ids=["host", "graph", "rank batches", "block tier"])
def test_union_parts_around_the_top_hub_count(opts):
    """Every graph of a disjoint union has its own top hubs: graphs just
    smaller and larger than the mask (256 hubs), tiny ones between them, and
    one dense enough for the block tier's hub maps."""
    gs = [G.chung_lu_graph(n, deg, 2.2, 40 + i)
          for i, (n, deg) in enumerate([(700, 6), (1, 2), (255, 8), (2, 2), (256, 8), (257, 8), (3000, 40), (33, 4)])]
    orders = [G.degree_order(g) for g in gs]
    sets = plb.build_batch([to_device(g, o) for g, o in zip(gs, orders)], plb.default_options(**opts))
    for i, (g, o) in enumerate(zip(gs, orders)):
        assert_labels_equal(sets[i], O.pll(g.off, g.col, o), f"part {i}")
