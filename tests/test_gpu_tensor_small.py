"""The tensor-core E-step on small problems, which the default path takes elsewhere: exact ties and duplicates, a lattice, no
distances wanted, scaling by powers of two, repeated runs, non-finite input, sizes around a tile, a chunk and a block, and a Lloyd loop in
lock step with the oracle.
"""
import numpy as np
import pytest
import torch

import oracle
from tests import gpu_util as u

pytestmark = pytest.mark.gpu


def _assign(X, C, **kw):
    from paper_2503_13089_b200 import binding as cc
    return u.gpu_assign(X, C, path=cc.PATH_TENSOR, **kw)


def _exact(X, C):
    idx, dist, obj, flagged, pts = _assign(X, C, want_flagged=True)
    want, d1 = oracle.assign(X, C)[:2]
    assert np.array_equal(idx, want) and np.array_equal(dist, d1.astype(np.float32))
    assert abs(obj - float(d1.astype(np.float32).astype(np.float64).sum())) <= len(X) * 2.0 ** -52 * obj
    assert len(set(pts.tolist())) == flagged <= len(X)
    return flagged


@pytest.mark.parametrize("N,g,K", [
    (1, 4, 1), (127, 1, 63), (128, 2, 64), (129, 3, 65), (1023, 4, 255), (1024, 5, 256), (1025, 6, 257), (2049, 7, 511), (300, 8, 513),
    (900, 9, 1000), (700, 12, 300), (513, 15, 129), (400, 16, 1025), (20000, 4, 700),
])
def test_sizes(N, g, K):
    rng = np.random.default_rng(N + g)
    X = (rng.standard_t(3.0, (N, g)) * 0.02).astype(np.float16)
    _exact(X, (rng.standard_normal((K, g)) * 0.03).astype(np.float32))


@pytest.mark.parametrize("g,K", [(1, 40), (4, 300), (7, 70), (8, 129), (16, 260)])
def test_ties_go_to_the_lowest_index(g, K):
    """Every centroid twice, points on a lattice: the near-ties and exact ties are all decided by the exact stage."""
    rng = np.random.default_rng(g)
    half = (rng.integers(-3, 4, ((K + 1) // 2, g)) / 4).astype(np.float32)
    C = np.concatenate([half, half])[:K]
    X = (rng.integers(-3, 4, (1500, g)) / 4).astype(np.float16)
    flagged = _exact(X, C)
    assert flagged >= 1500 * 0.9                        # the duplicate of the winner is as close


def test_without_distances_scaled_and_repeated():
    rng = np.random.default_rng(8)
    X = (rng.standard_normal((3000, 6)) * 0.5).astype(np.float16)
    C = (rng.standard_normal((500, 6)) * 0.5).astype(np.float32)
    idx, dist, obj, _ = _assign(X, C)
    assert np.array_equal(_assign(X, C, want_dist=False)[0], idx)
    again = _assign(X, C)
    assert np.array_equal(again[0], idx) and np.array_equal(again[1], dist) and again[2] == obj
    big = _assign((X * np.float16(16)).astype(np.float16), C * np.float32(16))       # exact in both types
    assert np.array_equal(big[0], idx) and np.array_equal(big[1], dist * np.float32(256))


def test_non_finite_input_is_reported():
    from paper_2503_13089_b200 import binding as cc
    X = np.ones((300, 4), dtype=np.float16)
    X[7, 2] = np.inf
    with pytest.raises(cc.CCError) as e:
        _assign(X, np.eye(4, dtype=np.float32))
    assert e.value.status == 8
    cc.cc_set_path(u.ctx(), cc.PATH_AUTO)


@pytest.mark.parametrize("N,g,K,iters", [(4000, 4, 100, 6), (3000, 7, 257, 4), (2000, 16, 64, 4)])
def test_fit_in_lock_step_with_the_oracle(N, g, K, iters):
    from paper_2503_13089_b200 import binding as cc
    rng = np.random.default_rng(N)
    X = (rng.standard_t(3.0, (N, g)) * 0.02).astype(np.float16)
    C0 = oracle.init_codebook(X, K, 5)
    C_or, idx_or, dist_or, counts_or, obj_or = oracle.fit(X, C0, iters)
    c = u.ctx()
    c.ensure_workspace(N, g, K)
    cc.cc_set_path(c, cc.PATH_TENSOR)
    C, idx, dist = u.dev(C0), torch.empty(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda")
    counts, trace = torch.empty(K, dtype=torch.int32, device="cuda"), torch.zeros(iters, dtype=torch.float64, device="cuda")
    cc.cc_fit(c, u.half_dev(X), N, g, K, iters, C, idx, dist, counts, trace)
    cc.cc_poll_status(c)
    cc.cc_set_path(c, cc.PATH_AUTO)
    assert np.array_equal(u.u16_np(idx).astype(np.int64), idx_or) and np.array_equal(counts.cpu().numpy(), counts_or)
    assert np.array_equal(C.cpu().numpy().view(np.uint32), C_or.view(np.uint32)) and np.array_equal(dist.cpu().numpy(), dist_or.astype(np.float32))
    assert np.allclose(trace.cpu().numpy(), obj_or, rtol=2.0 ** -24 + 2 * N * 2.0 ** -53, atol=0.0)
