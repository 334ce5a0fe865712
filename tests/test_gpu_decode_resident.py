"""Decode of many tiles with the codebook's head in shared memory: codebooks of one row, just inside and just outside what
fits, odd sizes, every row in use, ragged tiles on both edges; the same bits as numpy indexing."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,d_out,K", [
    (4, 8206, 1), (4, 8206, 3001), (4, 8206, 24703), (4, 8206, 24705), (4, 8206, 33001), (4, 8206, 65535),
    (8, 8203, 5), (8, 8203, 12351), (8, 8203, 12353), (8, 8203, 20001), (8, 8203, 65536),
    # short codebooks want more tiles
    (4, 16394, 1), (4, 16394, 3001), (4, 16394, 5999), (4, 8206, 5999), (4, 8206, 6000), (8, 16403, 5), (8, 16403, 5999), (8, 8203, 6001),
])
def test_decode_resident(g, d_out, K):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    d_in = 2568
    rng = np.random.default_rng(g * 7919 + K)
    N = cc.cc_num_subvectors(d_out, d_in, g, 0)
    C16 = rng.standard_normal((K, g)).astype(np.float16)
    idx = rng.integers(0, K, N).astype(np.uint16)
    idx[:K] = np.arange(K)[::-1].astype(np.uint16)     # every row is used
    What = torch.zeros((d_out, d_in), dtype=torch.float16, device="cuda")
    cc.cc_decode(u.ctx(), u.half_dev(C16), K, g, u.dev(idx.view(np.int16)).view(torch.uint16), d_out, d_in, 0, What)
    want = oracle.decode(C16, idx.astype(np.int32), d_out, d_in, 0)
    assert np.array_equal(u.u16_np(What.view(torch.uint16)).reshape(d_out, d_in), want.view(np.uint16))
