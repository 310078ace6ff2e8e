"""Graph mode: a segment starts with buffers that have room for its rounds (each
stop is another capture and instantiation, and there are eight of them)."""
import pytest

import oracle as O
from paper_1906_12018_gb300 import graphs as G

from gpu_util import assert_labels_equal, gpu_build

pytestmark = pytest.mark.gpu


def test_probe_index_with_room_for_a_segments_updates():
    """The pool of the probe index is sized for the tables as they are packed and
    for those that the segment's rounds outgrow: these rounds find room in it."""
    g = G.chung_lu_graph(2000, 2, 2.6, 1)
    order = G.degree_order(g)
    lab = gpu_build(g, order, use_graph=1)
    assert_labels_equal(lab, O.pll(g.off, g.col, order))
    assert lab.stats()["rounds"] > 8 and lab.stats()["reruns"] == 0


def test_small_frontiers_with_padded_rows():
    """The frontier buffers of a small graph hold 1,024 hubs however short their
    rows are (rows are padded to eight hubs).  The rounds of this graph bring
    fewer: its only stop is not one for their sake."""
    w = 10
    g = G.from_edges(w * w, [(w * i + j, w * i + j + 1) for i in range(w) for j in range(w - 1)] +
                     [(w * i + j, w * i + j + w) for i in range(w - 1) for j in range(w)])
    order = G.degree_order(g)
    lab = gpu_build(g, order, use_graph=1)
    assert_labels_equal(lab, O.pll(g.off, g.col, order))
    assert lab.stats()["reruns"] <= 1
