"""The pruned E-step (many points, many centroids) against the exhaustive one, which other tests hold against the oracle, and
against the oracle on a sample: the same codes, distances, counts, centroids and objectives in every iteration, whatever
the sizes around a tile of 128 points, a chunk of 64 centroids or a node of the tree, with ties, values far apart and
clusters that empty.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _points(N, g, K, kind):
    gen = torch.Generator(device="cuda").manual_seed(N + 7 * g + K)
    X = torch.randn((N, g), device="cuda", generator=gen)
    if kind == "heavy":
        X = X / torch.randn((N, 1), device="cuda", generator=gen).abs().clamp_(min=1e-3) * 0.02
        X[::4097] *= 3000.0
    elif kind == "ties":
        X = (X * 2).round() / 4                          # few distinct values: duplicates among points and centroids
    elif kind == "clumps":
        X = X * 1e-3 + torch.randint(-3, 4, (N, 1), device="cuda", generator=gen).float()
    return X.clamp_(-60000, 60000).to(torch.float16)


def _fit(X, g, K, iters, C0, path):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    c, N = u.ctx(), X.shape[0]
    cc.cc_set_path(c, path)
    C, idx, dist = C0.clone(), torch.empty(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda")
    counts, trace = torch.empty(K, dtype=torch.int32, device="cuda"), torch.zeros(iters, dtype=torch.float64, device="cuda")
    cc.cc_fit(c, X, N, g, K, iters, C, idx, dist, counts, trace)
    cc.cc_poll_status(c)
    cc.cc_set_path(c, cc.PATH_AUTO)
    return C, idx.view(torch.int16), dist, counts, trace


@pytest.mark.parametrize("N,g,K,iters,kind", [
    (2100001, 4, 4097, 17, "ties"), (1000003, 4, 16385, 4, "heavy"), (2000003, 3, 9001, 2, "heavy"), (400129, 6, 24003, 17, "clumps"),
    (2200000, 2, 4100, 5, "heavy"), (300031, 1, 30000, 5, "heavy"), (150001, 7, 65500, 17, "heavy"), (150000, 8, 65536, 17, "ties"),
    (524288, 5, 65535, 5, "heavy"), (140000, 6, 65535, 6, "ties"), (4000001, 4, 8193, 2, "clumps"), (2000003, 6, 61000, 5, "heavy"),
    (190001, 6, 65535, 6, "ties"), (4400001, 4, 8193, 2, "clumps"), (1990001, 3, 8200, 2, "heavy"),
])
def test_pruned_fit_equals_exhaustive_fit(N, g, K, iters, kind):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    c = u.ctx()
    c.ensure_workspace(N, g, K)
    X = _points(N, g, K, kind)
    C0 = torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(c, X, N, g, K, 3, C0)
    a = _fit(X, g, K, iters, C0, cc.PATH_AUTO)
    b = _fit(X, g, K, iters, C0, cc.PATH_TENSOR)
    for x, y in zip(a[:4], b[:4]):
        assert torch.equal(x, y)
    # the objectives are sums of the same FP32 distances, exact here and in a tree of FP64 additions there
    assert torch.allclose(a[4], b[4], rtol=2.0 ** -53 * 4096, atol=0.0)
    again = _fit(X, g, K, iters, C0, cc.PATH_AUTO)
    assert all(torch.equal(x, y) for x, y in zip(a, again))
    # one E-step by itself, without distances wanted, and its list of points decided exactly
    idx, n = torch.empty(N, dtype=torch.uint16, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
    cc.cc_assign(c, X, N, g, a[0], K, idx, None, None, n)
    flagged = u.last_flagged(N, g, K, int(n.item()))
    assert len(set(flagged.tolist())) == len(flagged) and (len(flagged) == 0 or (flagged.min() >= 0 and flagged.max() < N))
    rng = np.random.default_rng(K)
    sel = np.unique(np.concatenate([rng.integers(0, N, 60), flagged[:20], [0, N - 1]])).astype(np.int64)
    want = oracle.assign(X[torch.from_numpy(sel).cuda()].cpu().numpy(), a[0].cpu().numpy())[0]
    assert np.array_equal(u.u16_np(idx)[sel].astype(np.int64), want)


def test_objectives_of_a_longer_fit_start_with_those_of_a_shorter_one():
    """g = 8: fifteen iterations run exhaustively, sixteen in spatial order; the first objectives have the same bits."""
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    N, g, K = 150000, 8, 60001
    u.ctx().ensure_workspace(N, g, K)
    X = _points(N, g, K, "heavy")
    C0 = torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(u.ctx(), X, N, g, K, 1, C0)
    shorter, longer = _fit(X, g, K, 15, C0, cc.PATH_AUTO)[4], _fit(X, g, K, 16, C0, cc.PATH_AUTO)[4]
    assert torch.equal(shorter, longer[:15])


def test_pruned_non_finite_input_is_reported():
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    N, g, K = 600000, 4, 60000
    u.ctx().ensure_workspace(N, g, K)
    X = _points(N, g, K, "heavy")
    C0 = torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(u.ctx(), X, N, g, K, 1, C0)
    X[77, 1] = float("inf")
    with pytest.raises(cc.CCError) as e:
        _fit(X, g, K, 2, C0, cc.PATH_AUTO)
    assert e.value.status == 8
    cc.cc_set_path(u.ctx(), cc.PATH_AUTO)


def test_fit_in_the_smaller_workspace_gives_the_same():
    """cc_workspace_bytes is enough for every call; with cc_workspace_bytes_preferred the same fit may be pruned."""
    from paper_2503_13089_b200 import binding as cc
    N, g, K, iters = 1000003, 3, 9000, 5
    assert cc.cc_workspace_bytes_preferred(N, g, K) > cc.cc_workspace_bytes(N, g, K)
    assert cc.cc_workspace_bytes_preferred(N, 9, K) == cc.cc_workspace_bytes(N, 9, K)
    assert cc.cc_workspace_bytes_preferred(N, 17, K) == 0
    X = _points(N, g, K, "heavy")
    out = []
    for size in (cc.cc_workspace_bytes, cc.cc_workspace_bytes_preferred):
        c = cc.Context(0)
        ws = torch.empty(size(N, g, K), dtype=torch.uint8, device="cuda")
        cc.cc_set_workspace(c, ws, ws.numel())
        C = torch.empty((K, g), device="cuda")
        cc.cc_init_codebook(c, X, N, g, K, 3, C)
        idx, dist = torch.empty(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda")
        counts, trace = torch.empty(K, dtype=torch.int32, device="cuda"), torch.zeros(iters, dtype=torch.float64, device="cuda")
        before = cc.cc_launch_count(c)
        cc.cc_fit(c, X, N, g, K, iters, C, idx, dist, counts, trace)
        cc.cc_poll_status(c)
        out.append((C, idx.view(torch.int16), dist, counts, trace, cc.cc_launch_count(c) - before))
        torch.cuda.synchronize()
    assert out[0][5] != out[1][5]                        # two different ways
    assert all(torch.equal(x, y) for x, y in zip(out[0][:5], out[1][:5]))


@pytest.mark.parametrize("size", ["preferred", "needed"])
def test_an_undefined_point_is_infinitely_far_away(size):
    """Points that are not numbers have no nearest centroid; their distances and the objective are infinite whichever E-step ran,
    and the other points keep theirs."""
    from paper_2503_13089_b200 import binding as cc
    N, g, K = 600000, 4, 60000
    c = cc.Context(0)
    ws = torch.empty((cc.cc_workspace_bytes_preferred if size == "preferred" else cc.cc_workspace_bytes)(N, g, K), dtype=torch.uint8, device="cuda")
    cc.cc_set_workspace(c, ws, ws.numel())
    X = _points(N, g, K, "heavy")
    C = torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(c, X, N, g, K, 1, C)
    X[77, 1], X[N - 1, 3], X[4000, 0] = float("nan"), float("nan"), float("inf")
    out = {}
    for path in (cc.PATH_AUTO, cc.PATH_TENSOR):
        cc.cc_set_path(c, path)
        idx, dist = torch.empty(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda")
        obj = torch.zeros(1, dtype=torch.float64, device="cuda")
        cc.cc_assign(c, X, N, g, C, K, idx, dist, obj, None)
        with pytest.raises(cc.CCError):
            cc.cc_poll_status(c)
        assert obj.item() == float("inf") and torch.equal(torch.isinf(dist).nonzero().flatten().cpu(), torch.tensor([77, 4000, N - 1]))
        out[path] = (idx.view(torch.int16), dist)
    fine = torch.isfinite(out[cc.PATH_TENSOR][1])
    assert int(fine.sum()) == N - 3 and all(torch.equal(a[fine], b[fine]) for a, b in zip(out[cc.PATH_AUTO], out[cc.PATH_TENSOR]))
