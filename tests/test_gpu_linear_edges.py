"""The layer forward where a plan or a load meets its limit: codebooks whose slices end within a few rows of what shared memory
holds beside a full x, layers of few code groups, infinite activations, and workspaces that start on any 16-byte
boundary.  Same bound as in test_gpu_linear_paths: (d_in + 64) 2^-23 sum |x w|.
"""
import numpy as np
import pytest
import torch

from tests.test_gpu_linear_paths import _case, _run, _want

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,d_out,d_in,g,K", [
    (4, 14336, 2048, 4, 53700), (2, 11008, 2048, 8, 53696), (2, 11008, 2048, 8, 53700), (2, 8192, 2048, 7, 61380), (1, 11008, 4096, 7, 61385),
    (1, 11008, 4096, 7, 61376), (2, 11008, 4096, 8, 40280),
    # few code groups: either side of where the tensor kernel takes over
    (1, 1024, 4096, 16, 4096), (2, 1024, 4096, 16, 256), (1, 2048, 4096, 16, 256), (2, 512, 512, 16, 300), (2, 1024, 4096, 9, 20000),
    (4, 1024, 4096, 4, 65536), (2, 1024, 4096, 4, 65536), (3, 128, 4096, 4, 256), (1, 128, 4096, 2, 256),
])
def test_slices_and_layers_at_their_limits(M, d_out, d_in, g, K):
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, K)
    y, _ = _run(x, C16, idx, d_out, d_in, bias)
    want, bound = _want(x, C16, idx, d_out, d_in, bias)
    assert np.all(np.abs(y - want) <= bound), float(np.max(np.abs(y - want) / bound))


@pytest.mark.parametrize("M,d_out,d_in,g,K,q4", [
    (1, 4096, 2048, 4, 65536, False), (2, 520, 300, 6, 65500, False), (4, 260, 500, 4, 30000, False), (1, 130, 70, 9, 15000, False),
    (2, 300, 130, 4, 100, False), (2, 300, 130, 4, 3000, True), (9, 300, 200, 4, 3000, False), (200, 300, 200, 8, 3000, False),
])
def test_infinite_activations(M, d_out, d_in, g, K, q4):
    """y = x . w as IEEE arithmetic has it: +-infinity where one x is infinite and w is not zero, undefined where it is."""
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, 11)
    x[0, 7] = np.inf
    x[M - 1, d_in - 1] = -np.inf
    y, book = _run(x, C16, idx, d_out, d_in, bias, q4)
    with np.errstate(invalid="ignore"):
        want, _ = _want(np.where(np.isinf(x), 0, x).astype(np.float16), book, idx, d_out, d_in, bias)
        W = book[idx.astype(np.int64)].reshape(d_in, -1)[:, :d_out].astype(np.float64)
        for m, i in np.argwhere(np.isinf(x)):
            want[m] += float(x[m, i]) * W[i]
    odd = ~np.isfinite(want)
    assert np.array_equal(np.isnan(y), np.isnan(want)) and np.array_equal(y[odd & ~np.isnan(want)], want[odd & ~np.isnan(want)])
    assert odd[0].all() and np.isfinite(y[~odd]).all()


@pytest.mark.parametrize("M,d_out,d_in,g,K,q4", [
    (6, 1700, 4096, 16, 3000, False), (5, 2500, 4400, 9, 20001, False), (20, 3700, 3700, 11, 65536, False), (200, 4000, 4000, 13, 16000, False),
    (7, 3000, 3000, 6, 65536, False), (3, 4100, 4800, 16, 777, False), (1, 700, 900, 4, 60000, False), (2, 700, 900, 4, 60000, True), (300, 516, 260, 16, 16384, True),
])
@pytest.mark.parametrize("shift", [16, 48])
def test_workspace_on_a_16_byte_boundary(M, d_out, d_in, g, K, q4, shift):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, shift)
    c = cc.Context(0)
    room = torch.zeros(cc.cc_linear_workspace_bytes(c, M, d_out, d_in) + 64, dtype=torch.uint8, device="cuda")
    cc.cc_set_workspace(c, room[shift:], room.numel() - 64)
    book, codes, y = u.half_dev(C16), u.dev(idx.view(np.int16)).view(torch.uint16), torch.full((M, d_out), float("nan"), device="cuda")
    if q4:
        q, s, deq = torch.zeros((K * g + 1) // 2, dtype=torch.uint8, device="cuda"), torch.zeros(1, device="cuda"), torch.zeros((K, g), dtype=torch.float16, device="cuda")
        cc.cc_quantize_codebook(c, book, K, g, 4, q, s, deq)
        cc.cc_linear_forward_q4(c, u.half_dev(x), M, q, s, K, g, codes, d_out, d_in, u.dev(bias), y)
        C16 = deq.cpu().numpy()
    else:
        cc.cc_linear_forward(c, u.half_dev(x), M, book, K, g, codes, d_out, d_in, u.dev(bias), y)
    cc.cc_poll_status(c)
    want, bound = _want(x, C16, idx, d_out, d_in, bias)
    assert np.all(np.abs(y.cpu().numpy() - want) <= bound)
