"""The layer forward plane by plane at the edges of its tiles.  Bound: as in test_gpu_linear_paths (products exact, additions FP32)."""
import numpy as np
import pytest
import torch

from tests.test_gpu_linear_paths import _case, _run, _want
from tests.test_planes_plan import LAYERS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,d_out,d_in,g,K,q4", [
    # four, two and one coordinate a look-up; tokens around the operand's sizes; a last tile of one code group
    (5, 516, 640, 4, 16384, False), (16, 514, 1000, 4, 300, False), (17, 260, 257, 4, 20000, False), (64, 5000, 1700, 4, 65536, False),
    (65, 5000, 1700, 4, 65535, False), (128, 777, 900, 4, 3000, False), (192, 1026, 520, 6, 30001, False), (256, 1030, 530, 8, 32768, False),
    # an odd number of code groups (codes that start in the high half of a word), odd rows, planes that no coordinate fills
    (33, 655, 511, 5, 20000, False), (40, 1799, 333, 7, 16000, False), (12, 903, 640, 9, 32768, False), (30, 6600, 2048, 6, 65500, False),
    (7, 48, 700, 16, 12000, False), (250, 1040, 130, 13, 9, False), (20, 300, 4097, 1, 65536, False),
    # the 4-bit codebook
    (6, 500, 700, 4, 16384, True), (70, 1030, 640, 8, 32768, True), (64, 520, 515, 16, 12288, True),
])
def test_linear_planes(M, d_out, d_in, g, K, q4):
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, M + d_out + d_in + g)
    y, book = _run(x, C16, idx, d_out, d_in, bias, q4)
    want, bound = _want(x, book, idx, d_out, d_in, bias)
    assert np.all(np.abs(y - want) <= bound), float(np.max(np.abs(y - want) / bound))
    y2, _ = _run(x, C16, idx, d_out, d_in, bias, q4)
    assert np.array_equal(y.view(np.uint32), y2.view(np.uint32))


@pytest.mark.parametrize("M,d_out,d_in,g,K,q4", [layer for layer, _ in LAYERS])
def test_linear_planes_where_they_are_taken(M, d_out, d_in, g, K, q4):
    test_linear_planes(M, d_out, d_in, g, K, q4)


@pytest.mark.parametrize("M,d_out,d_in,g,K", [
    (33, 10000, 1300, 6, 65500), (200, 3000, 2760, 4, 65536),                # one coordinate a look-up; four and two stages
    (129, 793, 523, 2, 25467), (12, 903, 1300, 9, 3000),                     # two
    (26, 1085, 4491, 16, 19780), (91, 260, 2380, 16, 17185), (128, 777, 900, 4, 3000),  # four
])
def test_linear_planes_codes_off_a_word_boundary_and_least_workspace(M, d_out, d_in, g, K):
    """Codes that start on an odd address of 16-bit words, with the workspace of the preferred size; then with the smallest that the call
    accepts, where that is smaller the tensor kernel takes it: the same answer within the bound."""
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, 11)
    want, bound = _want(x, C16, idx, d_out, d_in, bias)
    room = torch.zeros(len(idx) + 1, dtype=torch.int16, device="cuda")
    room[1:] = torch.from_numpy(idx.view(np.int16)).cuda()
    xd, book, b, y = u.half_dev(x), u.half_dev(C16), u.dev(bias), torch.empty((M, d_out), device="cuda")
    ctx = cc.Context(0)
    need, most = cc.cc_linear_workspace_bytes(ctx, M, d_out, d_in), cc.cc_linear_workspace_bytes_preferred(ctx, M, d_out, d_in, g, K)
    assert need <= most
    ws = torch.zeros(most, dtype=torch.uint8, device="cuda")

    def run(codes, n):
        cc.cc_set_workspace(ctx, ws, n)
        y.fill_(float("nan"))
        cc.cc_linear_forward(ctx, xd, M, book, K, g, codes, d_out, d_in, b, y)
        cc.cc_poll_status(ctx)
        got = y.cpu().numpy()
        assert np.all(np.abs(got - want) <= bound)
        return got

    aligned = torch.from_numpy(idx.view(np.int16)).cuda().view(torch.uint16)
    by_planes = run(room.view(torch.uint16)[1:], most)
    assert np.array_equal(by_planes, run(aligned, most))                     # the same sums, however the codes lie
    least = run(room.view(torch.uint16)[1:], need)
    assert need == most or not np.array_equal(by_planes, least)              # another kernel, another order of the sums
    with pytest.raises(cc.CCError):
        run(aligned, need - 256)
    ctx.close()


def test_linear_workspace_sizes():
    """What every call needs, and what the planes take beside it: only where they take the call, and no more than their plan."""
    from paper_2503_13089_b200 import binding as cc
    ctx = cc.Context(0)
    for M, d_out, d_in, g, K, need, most in [(1, 4096, 4096, 4, 65536, 5.9, 5.9), (33, 1024, 1024, 4, 16000, 2.7, 4.3), (33, 11008, 4096, 6, 65500, 13.8, 20.3),
                                             (256, 8192, 28672, 4, 16000, 149, 252), (256, 8192, 28672, 6, 65500, 149, 149),
                                             (256, 28672, 8192, 4, 65536, 237, 242),
                                             (4096, 4096, 4096, 4, 65536, 539, 539)]:                # room for eight sets of partial sums
        a, b = cc.cc_linear_workspace_bytes(ctx, M, d_out, d_in), cc.cc_linear_workspace_bytes_preferred(ctx, M, d_out, d_in, g, K)
        assert a <= need * 1e6 and a <= b <= most * 1e6, (M, d_out, d_in, g, K, a, b)
    assert cc.cc_linear_workspace_bytes_preferred(ctx, 0, 8, 8, 4, 4) == cc.cc_linear_workspace_bytes_preferred(ctx, 1, 8, 8, 17, 4) == 0
    assert cc.cc_linear_workspace_bytes_preferred(ctx, 1, 8, 8, 4, 0) == cc.cc_linear_workspace_bytes_preferred(ctx, 1, 8, 8, 4, 65537) == 0
    ctx.close()
