"""Calls captured into a CUDA graph and replayed: launches that may begin before the one in front has ended, and the cooperative one
of the small fit.  The same bits as the call itself, on every replay."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _points(N, g, seed):
    from tests import gpu_util as u
    return u.half_dev((np.random.default_rng(seed).standard_t(3.0, (N, g)) * 0.02).astype(np.float16))


def _fit(N, g, K, iters):
    from paper_2503_13089_b200 import binding as cc
    c = cc.Context(0)
    c.ensure_workspace(N, g, K)
    X, C0 = _points(N, g, N + K), torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(c, X, N, g, K, 3, C0)
    out = [torch.empty_like(C0), torch.empty((K, g), dtype=torch.float16, device="cuda"), torch.empty(N, dtype=torch.int16, device="cuda"),
           torch.empty(N, device="cuda"), torch.empty(K, dtype=torch.int32, device="cuda"), torch.empty(iters + 1, dtype=torch.float64, device="cuda")]
    C, C16, idx, dist, counts, trace = out
    codes = idx.view(torch.uint16)

    def call():
        cc.cc_set_codebook(c, C0, K, g, C)
        cc.cc_fit(c, X, N, g, K, iters, C, codes, dist, counts, trace)
        cc.cc_finalize(c, X, N, g, C, K, C16, codes, dist, trace[iters:])
    return c, call, out


def _decode(d_out, d_in, g, K):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    c, rng = cc.Context(0), np.random.default_rng(d_out + g)
    C16 = u.half_dev(rng.standard_normal((K, g)).astype(np.float16))
    N = oracle.num_subvectors(d_out, d_in, g)
    codes = u.dev(rng.integers(0, K, N).astype(np.uint16).view(np.int16)).view(torch.uint16)
    W, X = torch.empty((d_out, d_in), dtype=torch.float16, device="cuda"), torch.empty((N, g), dtype=torch.float16, device="cuda")
    dC = torch.empty((K, g), device="cuda")
    c.ensure_workspace(N, g, K)

    def call():
        cc.cc_decode(c, C16, K, g, codes, d_out, d_in, cc.LAYOUT_PAPER_T, W)
        cc.cc_reshape_subvectors(c, W, d_out, d_in, g, cc.LAYOUT_PAPER_T, X)
        cc.cc_codebook_grad(c, X, N, g, codes, K, dC)
    return c, call, [W, X, dC]


def _linear(M, d_out, d_in, g, K, q4):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    from tests.test_gpu_linear_paths import _case
    c = cc.Context(0)
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, M + d_out)
    x, book, codes, b, y = u.half_dev(x), u.half_dev(C16), u.dev(idx.view(np.int16)).view(torch.uint16), u.dev(bias), torch.empty((M, d_out), device="cuda")
    c.ensure_workspace(1, g, K, at_least=cc.cc_linear_workspace_bytes_preferred(c, M, d_out, d_in, g, K))
    if not q4:
        return c, lambda: cc.cc_linear_forward(c, x, M, book, K, g, codes, d_out, d_in, b, y), [y]
    q, s = torch.zeros((K * g + 1) // 2, dtype=torch.uint8, device="cuda"), torch.zeros(1, device="cuda")
    cc.cc_quantize_codebook(c, book, K, g, 4, q, s)
    return c, lambda: cc.cc_linear_forward_q4(c, x, M, q, s, K, g, codes, d_out, d_in, b, y), [y]


@pytest.mark.parametrize("make,args", [
    (_fit, (5000, 4, 64, 4)), (_fit, (20000, 16, 200, 3)),                    # all iterations in one cooperative launch
    (_fit, (30000, 4, 2000, 3)), (_fit, (150000, 8, 1500, 2)),                # a launch an iteration; the tensor path
    (_fit, (1200000, 4, 8192, 3)),                                            # chunks ruled out
    (_decode, (2000, 2000, 5, 3000)), (_decode, (1024, 768, 4, 5000)), (_decode, (301, 77, 6, 100)),
    (_linear, (1, 1024, 1024, 4, 5000, False)), (_linear, (2, 1024, 1024, 8, 3000, True)),          # a few tokens
    (_linear, (12, 903, 1300, 9, 3000, False)), (_linear, (192, 1030, 1200, 4, 16384, True)),       # by planes
    (_linear, (8, 640, 1024, 16, 4000, False)), (_linear, (33, 3000, 2000, 6, 65500, False)),       # the tensor kernel, with a padded codebook
    (_linear, (300, 516, 260, 4, 300, False)),                                # the weight decoded once
])
def test_captured_and_replayed(make, args):
    from paper_2503_13089_b200 import binding as cc
    c, call, out = make(*args)

    def bits():
        cc.cc_poll_status(c)
        return [t.cpu().numpy().tobytes() for t in out]

    call()                                               # also sets what the kernels of this shape need once
    want = bits()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        call()
        call()                                           # back to back: the second begins while the first ends
    for _ in range(3):
        for t in out:
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert bits() == want
    graph.reset()
    c.close()
