"""The flat passes over arcs and label entries, and the prefix sums under them,
at the edges of their tiles (2,048 items), against the oracle (bit-exact)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1906_12018_gb300 import graphs as G
from paper_1906_12018_gb300 import plb

from gpu_util import assert_labels_equal, gpu_build, gpu_query

pytestmark = pytest.mark.gpu


def star_with_gaps(leaves, gap):
    """A star whose centre and leaves are separated by `gap` isolated vertices."""
    step = gap + 1
    return G.clean_csr(leaves * step + 1, np.zeros(leaves, np.int32),
                       (np.arange(1, leaves + 1) * step).astype(np.int32))


@pytest.mark.parametrize("leaves", [1, 1023, 1024, 1025, 2047, 2048, 2049, 4097])
@pytest.mark.parametrize("gap", [0, 1, 3])
def test_rows_at_tile_edges(leaves, gap):
    """Arc counts around one and two tiles; runs of empty rows inside a tile."""
    g = star_with_gaps(leaves, gap)
    order = G.degree_order(g)
    assert_labels_equal(gpu_build(g, order), O.pll(g.off, g.col, order))


@pytest.mark.parametrize("n", [2047, 2048, 2049, 4096, 4097, 70001])
def test_scans_at_tile_edges(n):
    """Vertex counts around one and two scan tiles, and many tiles."""
    g = G.chung_lu_graph(n, 4, 2.5, 3)
    order = G.degree_order(g)
    assert_labels_equal(gpu_build(g, order), O.pll(g.off, g.col, order))


@pytest.mark.parametrize("leaves", [8191, 8192, 8300])
def test_long_label_rows(leaves):
    """Rows around the length (8,192) from which a block instead of a warp
    merges and writes them: a star whose leaves all outrank its centre.  The
    i-th leaf is reached from the leaves before it over the centre alone, so it
    holds all of them at distance 2, and the centre holds every leaf."""
    g = star_with_gaps(leaves, 0)
    order = np.concatenate([np.arange(1, leaves + 1), [0]]).astype(np.int32)
    lab = gpu_build(g, order)
    off, hub, dist = lab.device_arrays()
    lens = torch.cat([torch.tensor([leaves + 1]), torch.arange(1, leaves + 1)]).cuda()
    assert torch.equal(off[1:] - off[:-1], lens)
    row = torch.repeat_interleave(torch.arange(leaves + 1, device="cuda"), lens)
    assert torch.equal(hub.long(), torch.arange(hub.numel(), device="cuda") - off[row])
    own = torch.zeros(hub.numel(), dtype=torch.bool, device="cuda")
    own[off[1:] - 1] = True
    assert torch.equal(dist.long(), torch.where(own, 0, torch.where(row == 0, 1, 2)))


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 4095, 4096, 4097, 8193, 70001])
@pytest.mark.parametrize("top", [0, 1, 255, 256, 70000, 1 << 24], ids=lambda t: f"deg{t}")
def test_degree_order_digits_and_tiles(n, top):
    """The radix sort at its tile edges, with degrees that vary in one, two,
    three or no bytes, many ties, and the bitonic path below it."""
    rng = np.random.default_rng(n + top)
    deg = rng.integers(0, top + 1, n) if top != 256 else rng.choice([0, 255, 256, 257], n)
    deg[rng.random(n) < 0.5] = min(top, 3)
    rp = torch.from_numpy(np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)).cuda()
    want = np.lexsort((np.arange(n), -deg)).astype(np.int32)
    assert np.array_equal(plb.degree_order(rp).cpu().numpy(), want)
    assert np.array_equal(plb.degree_order_noalloc(rp).cpu().numpy(), want)


@pytest.mark.parametrize("lens", [(1, 40), (31, 33), (32, 32), (33, 64), (65, 500), (127, 129)])
def test_queries_at_row_lengths(lens):
    """Rows around the 32 hubs that are compared in registers and the steps of
    the streamed part: stars whose centres are ranked last hold all their
    leaves, joined so that common hubs are found early, late or not at all."""
    edges, n = [], 0
    centres = []
    for k in lens + lens:  # two components of two stars each
        centres.append(n + k)
        edges += [(n + i, n + k) for i in range(k)]
        n += k + 1
    edges += [(0, lens[0] + 1), (centres[2] - 1, centres[3] - 1)]  # one pair joined at the top hubs, one at the last
    g = G.from_edges(n, edges)
    order = np.concatenate([np.setdiff1d(np.arange(n), centres), centres]).astype(np.int32)
    ref = O.pll(g.off, g.col, order)
    lab = gpu_build(g, order)
    pairs = np.stack(np.meshgrid(np.arange(n), centres + [0, n // 2]), -1).reshape(-1, 2).astype(np.int32)
    pairs = np.concatenate([pairs, pairs[:, ::-1]])
    assert np.array_equal(gpu_query(lab, pairs), O.query(ref, pairs))
