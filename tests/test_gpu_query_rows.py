"""Queries on rows around the lengths at which the query kernel changes its way
(up to 96 entries of the shorter row are all looked up; longer rows are bounded by
their first 32 hubs and streamed 128 entries at a time), with distances above 1,
against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1906_12018_gb300 import graphs as G
from paper_1906_12018_gb300 import plb

from gpu_util import gpu_build, gpu_query, to_device

pytestmark = pytest.mark.gpu


def spokes(parts, depth):
    """For each k of parts a centre with k chains of `depth` edges; returns the
    edges, the chain ends of each part and the centres.  With the ends ranked
    first and the centres next, a centre's row holds its k ends, at distance
    `depth`, and itself."""
    edges, ends, centres, n = [], [], [], 0
    for k in parts:
        first = n
        n += k
        mids = n + (depth - 1) * np.arange(k)
        n += (depth - 1) * k
        c, n = n, n + 1
        for i in range(k):
            chain = [first + i] + list(range(mids[i], mids[i] + depth - 1)) + [c]
            edges += list(zip(chain[:-1], chain[1:]))
        ends.append(np.arange(first, first + k))
        centres.append(c)
    return n, edges, ends, centres


@pytest.mark.parametrize("depth", [1, 2, 3])
@pytest.mark.parametrize("lens", [(94, 95), (95, 97), (96, 96), (97, 129), (126, 128), (160, 257)], ids=str)
def test_long_rows_of_far_hubs(lens, depth):
    """Four centres: two joined at an early hub over a detour and at their last
    hubs, two not joined at all."""
    n, edges, ends, centres = spokes(lens + lens, depth)
    edges += [(int(ends[0][0]), n), (n, n + 1), (n + 1, n + 2), (n + 2, int(ends[1][0]))]
    n += 3
    edges.append((int(ends[0][-1]), int(ends[1][-1])))
    g = G.from_edges(n, edges)
    top = np.concatenate(ends)
    rest = np.setdiff1d(np.arange(n), np.concatenate([top, centres]))
    order = np.concatenate([top, centres, rest]).astype(np.int32)
    ref = O.pll(g.off, g.col, order)
    assert np.diff(ref.off)[centres[2]] == lens[0] + 1
    lab = gpu_build(g, order)
    pairs = np.stack(np.meshgrid(np.arange(n), centres), -1).reshape(-1, 2).astype(np.int32)
    pairs = np.concatenate([pairs, pairs[:, ::-1]])
    assert np.array_equal(gpu_query(lab, pairs), O.query(ref, pairs))


@pytest.mark.parametrize("kind", ["unweighted", "weighted", "two parts"])
@pytest.mark.parametrize("seed", range(3))
def test_long_rows_of_random_orders(kind, seed):
    """Sparse random graphs in random order: rows of up to some hundred entries,
    whose common hubs lie anywhere."""
    rng = np.random.default_rng(seed)
    n = 1200
    s, t = rng.integers(0, n, 1700), rng.integers(0, n, 1700)
    if kind == "two parts":
        t = t // 2 * 2 + s % 2
    keep = s != t
    g = G.clean_csr(n, np.concatenate([s[keep], t[keep]]).astype(np.int32),
                    np.concatenate([t[keep], s[keep]]).astype(np.int32))
    order = rng.permutation(n).astype(np.int32)
    if kind == "weighted":
        wt = G.edge_weights(g, 1, 7, seed)
        ref = O.pll_weighted(g.off, g.col, wt, order)
        rp, col, o = to_device(g, order)
        lab = plb.build_weighted(rp, col, torch.from_numpy(wt).cuda(), o)
    else:
        ref = O.pll(g.off, g.col, order)
        lab = gpu_build(g, order)
    lens = np.diff(ref.off)
    assert np.sum(lens > 96) > 100 and np.sum(lens <= 96) > 100
    pairs = rng.integers(0, n, (200000, 2)).astype(np.int32)
    assert np.array_equal(gpu_query(lab, pairs), O.query(ref, pairs))
