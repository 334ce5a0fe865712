"""The layer forward's three ways through the GPU at the edges of their ranges: a few tokens (codes looked up in shared
memory, the FP16 codebook in slices), the tensor kernel with padded codebook rows, and many tokens (the weight decoded
once into tiles, then a product).

Bound: products of FP16 values are exact in FP32 and the additions are FP32.  An addition is off by at most 2^-23 of
the partial sum (the tensor core's own do not round to nearest), so an output is off by at most
(d_in + 64) 2^-23 sum |x w|; the 64 cover the additions of partial sums and the bias.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _case(M, d_out, d_in, g, K, seed):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal((M, d_in)) * 0.5).astype(np.float16)
    C16 = (rng.standard_t(3.0, (K, g)) * 0.02).astype(np.float16)
    idx = rng.integers(0, K, oracle.num_subvectors(d_out, d_in, g)).astype(np.uint16)
    idx[:min(len(idx), 2)] = K - 1                      # the last row of the codebook
    bias = rng.standard_normal(d_out).astype(np.float32)
    return x, C16, idx, bias


def _want(x, C16, idx, d_out, d_in, bias):
    g = C16.shape[1]
    W = C16[idx.astype(np.int64)].reshape(d_in, -1)[:, :d_out].astype(np.float64)
    x = x.astype(np.float64)
    return x @ W + bias, (d_in + 64) * 2.0 ** -23 * (np.abs(x) @ np.abs(W) + np.abs(bias))


def _run(x, C16, idx, d_out, d_in, bias, q4=False, off=0):
    """off: values by which the codebook's buffer is shifted from the start of an allocation."""
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    M, (K, g) = x.shape[0], C16.shape
    c = u.ctx()
    c.ensure_workspace(len(idx), g, K, at_least=cc.cc_linear_workspace_bytes_preferred(c, M, d_out, d_in, g, K))
    room = torch.full((off + K * g,), float("nan"), dtype=torch.float16, device="cuda")
    room[off:] = torch.from_numpy(C16.reshape(-1)).cuda()
    book, codes, y = room[off:], u.dev(idx.view(np.int16)).view(torch.uint16), torch.full((M, d_out), float("nan"), device="cuda")
    if q4:
        q, s, deq = torch.zeros((K * g + 1) // 2, dtype=torch.uint8, device="cuda"), torch.zeros(1, device="cuda"), torch.zeros((K, g), dtype=torch.float16, device="cuda")
        cc.cc_quantize_codebook(c, book, K, g, 4, q, s, deq)
        cc.cc_linear_forward_q4(c, u.half_dev(x), M, q, s, K, g, codes, d_out, d_in, u.dev(bias), y)
        C16 = deq.cpu().numpy()
    else:
        cc.cc_linear_forward(c, u.half_dev(x), M, book, K, g, codes, d_out, d_in, u.dev(bias), y)
    cc.cc_poll_status(c)
    return y.cpu().numpy(), C16


@pytest.mark.parametrize("M,d_out,d_in,g,K,q4,off", [
    # a few tokens: one slice, two and four; odd rows; a slice of one row; more in_features than one CTA takes
    (1, 300, 130, 4, 26000, False, 0), (2, 260, 70, 4, 26300, False, 0), (3, 264, 5000, 4, 65536, False, 0),
    (1, 130, 300, 7, 59999, False, 0), (2, 132, 300, 3, 33333, False, 8), (1, 75, 200, 9, 5001, False, 0),
    (1, 8192, 1024, 4, 3001, False, 0), (2, 6000, 1500, 4, 65535, False, 0),                # two groups a thread
    (4, 520, 4200, 4, 65536, True, 0), (2, 130, 777, 16, 16384, True, 0),
    # the tensor kernel: padded copy of the codebook, or none (few codes), and 16-value rows off a 32-byte boundary
    (5, 2000, 2000, 6, 5001, False, 0), (9, 2500, 900, 5, 20001, False, 8), (17, 250, 128, 5, 91, False, 0),
    (6, 260, 300, 16, 777, False, 8), (20, 4096, 1700, 16, 3000, False, 8), (33, 300, 96, 15, 19, False, 0),
    # many tokens: first and last size of a tile of tokens or out_features, in_features that end inside a tile, segments
    (192, 512, 512, 4, 300, False, 0), (193, 257, 511, 5, 301, False, 0), (255, 130, 1000, 7, 1001, False, 0),
    (257, 384, 2049, 8, 500, False, 0), (700, 129, 65, 16, 50, False, 8), (512, 1030, 130, 1, 9, False, 0),
    (96, 20000, 200, 9, 501, False, 0), (200, 700, 900, 6, 400, True, 0), (300, 516, 260, 16, 16384, True, 0),
    (8193, 136, 72, 2, 40, False, 0),                                                          # two passes over the tokens
])
def test_linear_paths(M, d_out, d_in, g, K, q4, off):
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, M + d_out + d_in + g)
    y, book = _run(x, C16, idx, d_out, d_in, bias, q4, off)
    want, bound = _want(x, book, idx, d_out, d_in, bias)
    assert np.all(np.abs(y - want) <= bound), float(np.max(np.abs(y - want) / bound))
    y2, _ = _run(x, C16, idx, d_out, d_in, bias, q4, off)
    assert np.array_equal(y.view(np.uint32), y2.view(np.uint32))


def test_linear_wide_in_panels():
    """A weight of more than 128 MB goes through the many-token path in panels of out_features; a sample of the columns."""
    M, d_out, d_in, g, K = 96, 17000, 4160, 8, 2000
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, 3)
    y, _ = _run(x, C16, idx, d_out, d_in, bias)
    assert np.isfinite(y).all()
    cols = np.concatenate([np.arange(0, 8), np.arange(8600, 8800), np.arange(d_out - 130, d_out)])
    W = C16[idx.astype(np.int64).reshape(d_in, -1)[:, cols // g], cols % g].astype(np.float64)
    x = x.astype(np.float64)
    err = np.abs(y[:, cols] - (x @ W + bias[cols]))
    assert np.all(err <= (d_in + 64) * 2.0 ** -23 * (np.abs(x) @ np.abs(W) + np.abs(bias[cols])))
