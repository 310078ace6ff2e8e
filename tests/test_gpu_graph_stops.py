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
