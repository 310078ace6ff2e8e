"""The candidate bounds up to which a receiver is left to a warp: 4 x 512 messages
with label rows of up to 128 entries, 2 x 512 with longer ones."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1906_12018_gb300 import graphs as G
from paper_1906_12018_gb300 import plb

from gpu_util import assert_labels_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hubs,senders,leaves,block", [
    (512, 2, 130, 0), (513, 2, 130, 1), (640, 2, 130, 1), (600, 2, 120, 0), (682, 3, 120, 0), (683, 3, 120, 1)])
def test_one_receiver(hubs, senders, leaves, block):
    """hubs -> senders -> v and leaves -> v: in round 2 only v receives, every hub
    from every sender, and L_in(v) holds the senders, the leaves and v.  Isolated
    vertices before them keep v's rank, the other limit of the bound, above it."""
    first = 4096
    v = first + hubs + senders + leaves
    a = np.arange(senders) + first + hubs
    src = np.concatenate([np.tile(np.arange(hubs) + first, senders), a, np.arange(leaves) + first + hubs + senders])
    dst = np.concatenate([np.repeat(a, hubs), np.full(senders + leaves, v)])
    g = G.directed_csr(v + 1, src.astype(np.int32), dst.astype(np.int32))
    order = np.arange(v + 1, dtype=np.int32)
    ref_in, ref_out = O.pll_directed(g.off, g.col, g.off_in, g.col_in, order)
    lin, lout = plb.build_directed(torch.from_numpy(g.off).cuda(), torch.from_numpy(g.col).cuda(),
                                   torch.from_numpy(order).cuda())
    assert_labels_equal(lin, ref_in)
    assert_labels_equal(lout, ref_out)
    assert lin.stats()["tier_vertices"][1] == block
