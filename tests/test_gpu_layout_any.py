"""Reshape and decode of rows that are no whole number of 16-byte pieces: every parity of row length and start, tiles with one
element over or missing, even and odd g, the last row of the codebook; the same bits as numpy transposes and indexing."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_out,d_in,g,K", [
    (64, 64, 6, 40), (65, 64, 6, 40), (63, 63, 7, 33), (1, 1, 1, 1), (130, 127, 5, 90), (127, 130, 3, 50), (66, 129, 2, 9),
    (200, 191, 4, 70), (321, 66, 9, 101), (97, 200, 10, 64), (129, 193, 13, 77), (1000, 777, 6, 3000), (515, 1024, 7, 65535),
    (259, 333, 16, 50), (258, 321, 8, 100), (300, 72, 15, 90), (127, 65, 12, 65),
])
def test_reshape_and_decode_any_row_length(d_out, d_in, g, K):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    rng = np.random.default_rng(d_out * 7 + d_in + g)
    W = rng.standard_normal((d_out, d_in)).astype(np.float16)
    N = cc.cc_num_subvectors(d_out, d_in, g, 0)
    X = torch.full((N * g + 64,), 7.0, dtype=torch.float16, device="cuda")
    cc.cc_reshape_subvectors(u.ctx(), u.half_dev(W), d_out, d_in, g, 0, X)
    got = u.u16_np(X.view(torch.uint16))
    assert np.array_equal(got[:N * g].reshape(N, g), oracle.reshape_subvectors(W, g).view(np.uint16))
    assert np.all(got[N * g:] == np.float16(7.0).view(np.uint16))               # nothing behind the end
    C16 = rng.standard_normal((K, g)).astype(np.float16)
    idx = rng.integers(0, K, N).astype(np.uint16)
    idx[:2] = K - 1
    What = torch.full((d_out * d_in + 64,), 7.0, dtype=torch.float16, device="cuda")
    cc.cc_decode(u.ctx(), u.half_dev(C16), K, g, u.dev(idx.view(np.int16)).view(torch.uint16), d_out, d_in, 0, What)
    got = u.u16_np(What.view(torch.uint16))
    assert np.array_equal(got[:d_out * d_in].reshape(d_out, d_in), oracle.decode(C16, idx.astype(np.int32), d_out, d_in, 0).view(np.uint16))
    assert np.all(got[d_out * d_in:] == np.float16(7.0).view(np.uint16))
