"""Small problems (one launch an iteration): sizes around a block, a group, a chunk of 32 centroids and the table's limit,
odd g, ties, emptied clusters and large values, against the oracle's free-running fit and exhaustive assignment.

Codes, counts, centroids and distances have one right answer.  The objective is the FP64 sum of the FP32 distances in
another order: off by at most N 2^-53 of itself and one FP32 rounding of each non-negative term.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,g,K,iters", [
    (1, 4, 1, 2), (5, 3, 5, 2), (255, 4, 31, 4), (256, 4, 32, 4), (257, 4, 33, 4), (1023, 1, 9, 3), (3001, 2, 64, 4),
    (9000, 5, 65, 3), (4000, 6, 1025, 3), (5000, 7, 100, 3), (2500, 8, 1500, 3), (3000, 9, 257, 3), (2000, 16, 1536, 2),
    (1700, 15, 300, 3), (38000, 4, 200, 3), (80001, 4, 130, 2), (7000, 4, 6144, 2),
    # few clusters, many points: either side of where the sums have a kernel of their own
    (40000, 16, 1, 2), (100001, 3, 1, 2), (250001, 8, 2, 3), (250000, 1, 64, 3), (260000, 2, 33, 3), (250003, 3, 8, 3),
])
def test_small_fit_matches_oracle(N, g, K, iters):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    rng = np.random.default_rng(N * 31 + g)
    X = (rng.standard_t(3.0, (N, g)) * 0.02).astype(np.float16)
    X[::7] = X[0]                                       # ties between equal centroids, clusters left empty
    X[3::11] = (rng.standard_normal((len(X[3::11]), g)) * 200).astype(np.float16)
    C0 = oracle.init_codebook(X, K, 5)
    C_or, idx_or, dist_or, counts_or, obj_or = oracle.fit(X, C0, iters)
    c = u.ctx()
    c.ensure_workspace(N, g, K)
    C, Xd = u.dev(C0), u.half_dev(X)
    idx, dist = torch.empty(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda")
    counts, trace = torch.empty(K, dtype=torch.int32, device="cuda"), torch.zeros(iters, dtype=torch.float64, device="cuda")
    cc.cc_fit(c, Xd, N, g, K, iters, C, idx, dist, counts, trace)
    cc.cc_poll_status(c)
    assert np.array_equal(u.u16_np(idx).astype(np.int64), idx_or) and np.array_equal(counts.cpu().numpy(), counts_or)
    assert np.array_equal(dist.cpu().numpy(), dist_or.astype(np.float32))
    assert np.array_equal(C.cpu().numpy().view(np.uint32), C_or.view(np.uint32))
    assert np.allclose(trace.cpu().numpy(), obj_or, rtol=2.0 ** -24 + 2 * N * 2.0 ** -53, atol=0.0)
    idx_a, dist_a, obj_a, flagged, pts = u.gpu_assign(X, C_or, want_flagged=True)
    idx_w, d1_w = oracle.assign(X, C_or)[:2]
    assert np.array_equal(idx_a, idx_w) and np.array_equal(dist_a, d1_w.astype(np.float32))
    assert len(set(pts.tolist())) == flagged <= N
