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


@pytest.mark.parametrize("lead", [0, 230, 16384 - 40, 32768 - 40, 147456 - 40, 147456 + 10])
@pytest.mark.parametrize("opts", [{}, {"use_graph": 1},
                                  {"warp_cand_cap": 32, "warp_label_cap": 16, "block_cand_cap": 64,
                                   "block_label_cap": 24, "block_threads": 64}], ids=["host", "graph", "block tier"])
@pytest.mark.parametrize("n,deg", [(2500, 40), (1500, 400)], ids=["sparse", "dense"])
def test_hubs_around_the_map_boundaries(n, deg, lead, opts):
    """The highest-ranked hubs are marked in byte maps and bitmaps, the others
    go into hash sets.  `lead` isolated vertices ranked first move a small
    graph's hubs to the boundaries: the top-hub masks (256), the block tier's
    byte map (16,384) and bitmap (147,456), the warp tier's bitmap (32,768)."""
    core = G.chung_lu_graph(n, deg, 2.2, 9)
    src = np.repeat(np.arange(core.n), np.diff(core.off))
    g = G.clean_csr(core.n + lead, src.astype(np.int32) + lead, core.col.astype(np.int32) + lead)
    order = np.concatenate([np.arange(lead, dtype=np.int32), G.degree_order(core) + np.int32(lead)])
    rp, col, o = to_device(g, order)
    lab = plb.build(rp, col, o, **opts)
    assert_labels_equal(lab, O.pll(g.off, g.col, order), f"lead {lead}")
    if lead > 4096 and deg == 400:  # (with few ranks the candidate bounds stay within the warp tier)
        assert lab.stats()["tier_vertices"][1] > 0
