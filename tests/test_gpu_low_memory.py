"""cc_compress_host where device memory does not reach to the preferred size: the same results in what every call needs, and the
buffer kept from then on."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_compress_keeps_its_buffer_when_memory_is_short():
    from paper_2503_13089_b200 import binding as cc
    d_out, d_in, g, K, iters = 8192, 8192, 4, 65536, 0
    N = cc.cc_num_subvectors(d_out, d_in, g, 0)
    extra = cc.cc_workspace_bytes_preferred(N, g, K) - cc.cc_workspace_bytes(N, g, K)
    assert extra > 2 << 30                              # room to be short of
    rng = np.random.default_rng(5)
    W = torch.from_numpy((rng.standard_normal((d_out, d_in), dtype=np.float32) * 0.02).astype(np.float16))
    C16, idx = torch.empty((K, g), dtype=torch.float16), torch.empty(N, dtype=torch.uint16)

    def call(c):
        cc.cc_compress_host(c, W, d_out, d_in, g, K, iters, 1, 0, C16, idx, None, None)
        return C16.clone(), idx.view(torch.int16).clone()

    want = call(cc.Context(0))                          # its context is gone: the buffer is given back
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    c = cc.Context(0)
    taken = 2 * d_out * d_in * 2 + N * 8 + cc.cc_workspace_bytes(N, g, K)       # about what the call needs
    ballast = torch.empty(torch.cuda.mem_get_info()[0] - taken - extra // 2, dtype=torch.uint8, device="cuda")
    got = call(c)
    assert all(torch.equal(a, b) for a, b in zip(want, got))
    kept = torch.cuda.mem_get_info()[0]
    call(c)
    assert torch.cuda.mem_get_info()[0] == kept
    del ballast
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    got = call(c)
    assert torch.cuda.mem_get_info()[0] == free and all(torch.equal(a, b) for a, b in zip(want, got))
