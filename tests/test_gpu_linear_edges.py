"""The layer forward where a plan or a load meets its limit: codebooks whose slices end within a few rows of what shared memory
holds beside a full x, and infinite activations.  Same bound as in test_gpu_linear_paths: (d_in + 64) 2^-23 sum |x w|.
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
