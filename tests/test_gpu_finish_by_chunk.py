"""The E-step's finish that takes a warp's points chunk by chunk (few centroids) against the direct FP32 path: both decide as the FP64
distances do, so codes and distances have the same bits, also for ties and doubled centroids."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,g,K", [
    (1, 4, 1), (31, 4, 63), (33, 4, 64), (1000, 4, 65), (40000, 4, 512), (40000, 4, 513), (5003, 1, 200), (20000, 5, 1024), (20001, 8, 1000), (9999, 16, 257),
    (5001, 3, 128), (5001, 3, 129), (5001, 2, 64), (7000, 13, 768), (7000, 15, 769), (9999, 16, 384), (9999, 16, 385),           # where the rule changes
])
def test_finish_by_chunk(N, g, K):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    rng = np.random.default_rng(N + g + K)
    X = rng.standard_t(3.0, (N, g)).astype(np.float16)
    C = rng.standard_t(3.0, (K, g)).astype(np.float32)
    C[K // 2:] = np.where(rng.random((K - K // 2, 1)) < 0.2, C[:K - K // 2], C[K // 2:])     # doubled centroids: ties
    X[: N // 8] = C[rng.integers(0, K, N // 8)].astype(np.float16)                            # points near or on a centroid
    Xd, Cd, c, got = u.half_dev(X), u.dev(C), u.ctx(), []
    c.ensure_workspace(N, g, K)
    try:
        for path in (cc.PATH_TENSOR, cc.PATH_FFMA):
            cc.cc_set_path(c, path)
            idx, dist = torch.zeros(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda")
            obj = torch.empty(1, dtype=torch.float64, device="cuda")
            cc.cc_assign(c, Xd, N, g, Cd, K, idx, dist, obj)
            cc.cc_poll_status(c)
            got.append((idx.cpu().numpy().tobytes(), dist.cpu().numpy().tobytes()))
    finally:
        cc.cc_set_path(c, cc.PATH_AUTO)
    assert got[0] == got[1]
