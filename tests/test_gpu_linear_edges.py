"""The layer forward where a plan or a load meets its limit: codebooks whose slices end within a few rows of what shared memory
holds beside a full x.  Same bound as in test_gpu_linear_paths: (d_in + 64) 2^-23 sum |x w|.
"""
import numpy as np
import pytest

from tests.test_gpu_linear_paths import _case, _run, _want

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,d_out,d_in,g,K", [
    (4, 14336, 2048, 4, 53700), (2, 11008, 2048, 8, 53696), (2, 11008, 2048, 8, 53700), (2, 8192, 2048, 7, 61380), (1, 11008, 4096, 7, 61385),
    (1, 11008, 4096, 7, 61376), (2, 11008, 4096, 8, 40280),
])
def test_slices_that_fill_shared_memory(M, d_out, d_in, g, K):
    x, C16, idx, bias = _case(M, d_out, d_in, g, K, K)
    y, _ = _run(x, C16, idx, d_out, d_in, bias)
    want, bound = _want(x, C16, idx, d_out, d_in, bias)
    assert np.all(np.abs(y - want) <= bound), float(np.max(np.abs(y - want) / bound))
