"""All iterations of a small fit in one launch against the same iterations one launch each: the same bits."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,g,K,iters", [
    (1, 3, 1, 3), (255, 4, 7, 4), (257, 4, 256, 5), (32768, 4, 1024, 7),          # one block, two, every block one step; K g at the bound
    (120000, 4, 257, 3), (70001, 1, 300, 6), (5000, 16, 256, 2),                  # several steps a block; odd sizes; long sub-vectors
])
def test_small_fit_in_one_launch(N, g, K, iters):
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    rng = np.random.default_rng(N + g + K)
    X = u.half_dev(rng.standard_t(3.0, (N, g)).astype(np.float16))
    c = u.ctx()
    c.ensure_workspace(N, g, K)
    C0 = torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(c, X, N, g, K, 5, C0)

    def buffers():
        return (C0.clone(), torch.zeros(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda"),
                torch.empty(K, dtype=torch.int32, device="cuda"), torch.zeros(iters, dtype=torch.float64, device="cuda"))

    a, b = buffers(), buffers()
    cc.cc_fit(c, X, N, g, K, iters, *a)
    for it in range(iters):
        cc.cc_fit(c, X, N, g, K, 1, *b[:4], b[4][it:])
    cc.cc_poll_status(c)
    for x, y in zip(a, b):
        assert x.cpu().numpy().tobytes() == y.cpu().numpy().tobytes()


def _fit(c, X, C0, iters):
    from paper_2503_13089_b200 import binding as cc
    (N, g), K = X.shape, C0.shape[0]
    out = (C0.clone(), torch.zeros(N, dtype=torch.uint16, device="cuda"), torch.empty(N, device="cuda"),
           torch.empty(K, dtype=torch.int32, device="cuda"), torch.zeros(iters, dtype=torch.float64, device="cuda"))
    cc.cc_fit(c, X, N, g, K, iters, *out)
    cc.cc_poll_status(c)
    return [t.cpu().numpy().tobytes() for t in out]


def test_small_fit_whatever_the_workspace_holds_and_after_a_time_out():
    """A fit depends on nothing in the workspace but its status block, in which it leaves the counters of other calls alone and its own
    at zero; a poll that reports a time-out leaves that block as cc_set_workspace does, whatever arrived after a kernel gave up."""
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    N, g, K, iters = 30000, 4, 300, 5
    rng = np.random.default_rng(17)
    X = u.half_dev(rng.standard_t(3.0, (N, g)).astype(np.float16))
    c = cc.Context(0)
    ws = torch.zeros(cc.cc_workspace_bytes(N, g, K), dtype=torch.uint8, device="cuda")
    cc.cc_set_workspace(c, ws, ws.numel())
    C0 = torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(c, X, N, g, K, 5, C0)
    want = _fit(c, X, C0, iters)
    words = ws[:4096].view(torch.int32)
    ws[4096:] = 255
    assert _fit(c, X, C0, iters) == want
    assert not words.any()
    words[64:] = 1                                       # the layer forward's counters
    assert _fit(c, X, C0, iters) == want
    assert (words[64:] == 1).all() and not words[40:64].any()
    words[0], words[8], words[56], words[57] = 2, 1, 1, 3  # the time-out's bit, a ticket that nobody took back, late arrivals
    with pytest.raises(cc.CCError) as e:
        cc.cc_poll_status(c)
    assert e.value.status == 9 and not ws[:4096].any()
    cc.cc_poll_status(c)
    assert _fit(c, X, C0, iters) == want
    c.close()


def test_small_fit_where_the_cooperative_launch_is_refused():
    """With more blocks than the device holds at once (a context that takes it to have 5000 SMs) the launch of all iterations is
    refused; the fit then runs one launch an iteration.  Codes, centroids, counts and distances are the same bits; the objective is
    summed over other blocks (float64, 3 10^5 positive terms: relative difference below 10^-10)."""
    import ctypes as ct
    from paper_2503_13089_b200 import binding as cc
    from tests import gpu_util as u
    N, g, K, iters = 300000, 4, 8, 4
    rng = np.random.default_rng(23)
    X = u.half_dev(rng.standard_t(3.0, (N, g)).astype(np.float16))
    c = cc.Context(0)
    c.ensure_workspace(N, g, K)
    C0 = torch.empty((K, g), device="cuda")
    cc.cc_init_codebook(c, X, N, g, K, 5, C0)
    want = _fit(c, X, C0, iters)
    n0 = cc.cc_launch_count(c)
    _fit(c, X, C0, iters)
    assert cc.cc_launch_count(c) - n0 == 1
    fields = (ct.c_int * 2).from_address(c._h.value)     # cc_ctx begins with the device and its number of SMs
    assert fields[0] == 0 and fields[1] == torch.cuda.get_device_properties(0).multi_processor_count
    fields[1] = 5000
    n0 = cc.cc_launch_count(c)
    got = _fit(c, X, C0, iters)
    assert cc.cc_launch_count(c) - n0 == iters
    assert got[:4] == want[:4]
    assert np.allclose(np.frombuffer(got[4]), np.frombuffer(want[4]), rtol=1e-10, atol=0.0)
    c.close()
