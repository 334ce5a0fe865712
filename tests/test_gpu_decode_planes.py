"""Decode by coordinates (rows of an odd number of values, large matrices) against a plain gather; bytes, so exact."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_out,d_in,g,K,off", [
    (1733, 1736, 5, 3000, 0), (1735, 1736, 5, 37376, 0), (2304, 1320, 9, 1, 0), (3001, 1000, 7, 16001, 0), (1750, 2008, 7, 999, 1), (1760, 1800, 15, 65, 1),
    (37000, 88, 11, 2000, 0), (12, 260000, 13, 300, 0),
    (2401, 1736, 5, 37376, 0), (3001, 1880, 7, 16001, 0), (3001, 1808, 7, 16001, 0), (2000, 1600, 11, 4000, 1), (2000, 1592, 11, 4000, 1),   # on both sides of the bound
])
def test_decode_planes(d_out, d_in, g, K, off):
    """off: codes that start on an odd address of 16-bit words."""
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    rng = np.random.default_rng(d_out + d_in + g)
    groups = -(-d_out // g)
    idx = rng.integers(0, K, (d_in, groups)).astype(np.uint16)
    idx[-1, -1] = K - 1
    C16 = rng.standard_normal((K, g)).astype(np.float16)
    room = torch.zeros(idx.size + off, dtype=torch.int16, device="cuda")
    room[off:] = torch.from_numpy(idx.reshape(-1).view(np.int16)).cuda()
    W = torch.full((d_out, d_in), float("nan"), dtype=torch.float16, device="cuda")
    cc.cc_decode(u.ctx(), u.half_dev(C16), K, g, room.view(torch.uint16)[off:], d_out, d_in, cc.LAYOUT_PAPER_T, W)
    want = C16[idx.astype(np.int64)].reshape(d_in, groups * g)[:, :d_out].T
    assert np.array_equal(W.cpu().numpy().view(np.uint16), np.ascontiguousarray(want).view(np.uint16))
