"""The flat passes over arcs and label entries, and the prefix sums under them,
at the edges of their tiles (2,048 items), against the oracle (bit-exact)."""
import numpy as np
import pytest

import oracle as O
from paper_1906_12018_gb300 import graphs as G

from gpu_util import assert_labels_equal, gpu_build

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
