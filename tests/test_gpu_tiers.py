"""The gather + prune tiers at the edges of their tables and masks, against the
oracle (bit-exact)."""
import numpy as np
import pytest
import torch

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
    """The highest-ranked hubs are marked in bitmaps, the others go into hash
    sets.  `lead` isolated vertices ranked first move a small graph's hubs to
    the boundaries: the top-hub masks (256), the block tier's bitmap (147,456),
    the warp tier's (32,768), and a rank between."""
    core = G.chung_lu_graph(n, deg, 2.2, 9)
    src = np.repeat(np.arange(core.n), np.diff(core.off))
    g = G.clean_csr(core.n + lead, src.astype(np.int32) + lead, core.col.astype(np.int32) + lead)
    order = np.concatenate([np.arange(lead, dtype=np.int32), G.degree_order(core) + np.int32(lead)])
    rp, col, o = to_device(g, order)
    lab = plb.build(rp, col, o, **opts)
    assert_labels_equal(lab, O.pll(g.off, g.col, order), f"lead {lead}")
    if lead > 4096 and deg == 400:  # (with few ranks the candidate bounds stay within the warp tier)
        assert lab.stats()["tier_vertices"][1] > 0


@pytest.mark.parametrize("lead", [0, 32768 - 700, 32768 - 300], ids=["bitmap", "both", "set"])
@pytest.mark.parametrize("opts", [{}, {"use_graph": 1}, {"warp_cand_cap": 32}], ids=["host", "graph", "small"])
def test_candidate_counts_around_the_warp_tiers_list(opts, lead):
    """Receivers of k candidates each, none with a witness, around the
    capacity of the warp tier's list (968, and 64 for the smallest option) and
    the bounds up to which it is tried: `lead` ranks before the hubs move all but the
    first of them past the bitmap (32,768), where the set holds 512 and 32."""
    counts = [31, 32, 33, 63, 64, 65, 80, 81, 128, 129, 512, 513, 967, 968, 969, 1024, 1025, 1280, 1281, 2048, 2049]
    hubs, senders = 2049, 16
    src, dst = [], []
    for q, k in enumerate(counts):
        v = hubs + len(counts) * senders + q
        for s in range(senders):
            a = hubs + senders * q + s
            mine = np.arange(s, k, senders)
            src += [mine, [a]]
            dst += [np.full(len(mine), a), [v]]
    n = lead + hubs + len(counts) * (senders + 1)
    g = G.clean_csr(n, (np.concatenate(src) + lead).astype(np.int32), (np.concatenate(dst) + lead).astype(np.int32))
    order = np.arange(n, dtype=np.int32)
    rp, col, o = to_device(g, order)
    lab = plb.build(rp, col, o, **opts)
    assert_labels_equal(lab, O.pll(g.off, g.col, order), f"lead {lead}")


@pytest.mark.parametrize("lead", [0, 40, 147456 - 1000], ids=["map", "offset", "map and set"])
def test_profiled_counts_agree_between_the_tiers(lead):
    """A profiled build counts the label entries below and of every checked
    candidate: the warp tier one candidate at a time, the block tier 64 hubs of
    its bitmap at a time."""
    core = G.chung_lu_graph(1800, 60, 2.2, 11)
    src = np.repeat(np.arange(core.n), np.diff(core.off))
    g = G.clean_csr(core.n + lead, src.astype(np.int32) + lead, core.col.astype(np.int32) + lead)
    order = np.concatenate([np.arange(lead, dtype=np.int32), G.degree_order(core) + np.int32(lead)])
    rp, col, o = to_device(g, order)
    warp = plb.build(rp, col, o, profile=1, warp_cand_cap=2048, warp_label_cap=512).stats()
    block = plb.build(rp, col, o, profile=1, warp_cand_cap=32, warp_label_cap=16).stats()
    assert block["tier_vertices"][1] > warp["tier_vertices"][1]
    for key in ("check_lv_entries", "check_lh_entries"):
        assert warp[key] == block[key] > 0, key


def hub_edges(leaves, arcs, seed):
    """Hubs 0..len(arcs)-1 with the given numbers of random leaves, and a sparse
    random graph on the leaves."""
    rng = np.random.default_rng(seed)
    k = len(arcs)
    src = [np.full(c, i) for i, c in enumerate(arcs)] + [k + rng.integers(0, leaves, leaves)]
    dst = [k + rng.choice(leaves, c, replace=False) for c in arcs] + [k + rng.integers(0, leaves, leaves)]
    return k + leaves, np.concatenate(src), np.concatenate(dst)


# arcs per hub: at and next to the least number that is split (2,048) and whole
# and ragged numbers of parts (1,024); the leaves' graph adds none to the hubs
HUB_ARCS = [2047, 2048, 2049, 3072, 3073, 5000, 9000]


@pytest.mark.parametrize("opts", [{}, {"use_graph": 1}, {"batch_hubs": 5000}], ids=["host", "graph", "rank batches"])
def test_split_receivers(opts):
    n, src, dst = hub_edges(9500, HUB_ARCS, 1)
    g = G.clean_csr(n, src.astype(np.int32), dst.astype(np.int32))
    rng = np.random.default_rng(2)
    mixed = rng.permutation(n).astype(np.int32)  # hubs anywhere in the order
    for order in (G.degree_order(g), mixed if not opts else None):
        if order is None:
            continue
        rp, col, o = to_device(g, order)
        assert_labels_equal(plb.build(rp, col, o, **opts), O.pll(g.off, g.col, order))


def test_split_receivers_weighted():
    n, src, dst = hub_edges(9500, HUB_ARCS, 3)
    g = G.clean_csr(n, src.astype(np.int32), dst.astype(np.int32))
    order = G.degree_order(g)
    wt = G.edge_weights(g, 1, 5, 4)
    rp, col, o = to_device(g, order)
    lab = plb.build_weighted(rp, col, torch.from_numpy(wt).cuda(), o)
    assert_labels_equal(lab, O.pll_weighted(g.off, g.col, wt, order))


def test_split_receivers_directed():
    n, src, dst = hub_edges(9500, HUB_ARCS, 5)
    flip = np.random.default_rng(6).random(src.size) < 0.4
    g = G.directed_csr(n, np.where(flip, dst, src), np.where(flip, src, dst))
    order = G.directed_degree_order(g)
    ref_in, ref_out = O.pll_directed(g.off, g.col, g.off_in, g.col_in, order)
    lin, lout = plb.build_directed(torch.from_numpy(g.off).cuda(), torch.from_numpy(g.col).cuda(),
                                   torch.from_numpy(order).cuda())
    assert_labels_equal(lin, ref_in, "in")
    assert_labels_equal(lout, ref_out, "out")
