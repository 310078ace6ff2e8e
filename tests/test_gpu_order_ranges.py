"""The degree order around the size where it turns from the bitonic network to the
radix sort."""
import numpy as np
import pytest
import torch

from paper_1906_12018_gb300 import plb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2049, 4096, 4097, 6000, 8191, 8192, 8193, 12289])
def test_order_and_its_scratch(n):
    """Small orders are latency: up to 8,192 vertices the network over keys padded
    to a power of two (8 bytes each, nothing else) is the faster one."""
    rng = np.random.default_rng(n)
    deg = np.minimum(rng.zipf(1.8, n), n)
    rp = torch.from_numpy(np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)).cuda()
    want = np.lexsort((np.arange(n), -deg)).astype(np.int32)
    torch.cuda.synchronize()
    before = plb.memory_stats(reset=True)["used"]
    got = plb.degree_order(rp)
    torch.cuda.synchronize()
    scratch = plb.memory_stats()["used_high"] - before
    assert np.array_equal(got.cpu().numpy(), want)
    if n <= 8192:
        assert scratch <= 8 * (1 << (n - 1).bit_length())
