"""The float32 SSE of 32 attributes in register tiles: 24 attributes with eight zero columns between
them have the same distances bit for bit, so labels and sums equal those of the 24 alone, which one
thread per row scores."""
import numpy as np
import pytest

from tests.test_gpu_wide_rows import _noalloc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 6, 255, 257, 2048, 2049, 30000])
@pytest.mark.parametrize("k", [23, 24, 25, 64, 65, 340])
def test_tiles_of_32_attributes(n, k):
    r = np.random.default_rng(n * 7 + k)
    x, c = r.random((n, 24), dtype=np.float32), r.random((k, 24), dtype=np.float32)
    c[k // 2] = c[0]                               # equal distances: the lower index
    at = np.sort(r.choice(32, 24, replace=False))
    y, e = np.zeros((n, 32), np.float32), np.zeros((k, 32), np.float32)
    y[:, at], e[:, at] = x, c
    want = _noalloc(x, c, 0)
    for off in (0, 1):
        got = _noalloc(y, e, off)
        np.testing.assert_array_equal(got[0], want[0])
        np.testing.assert_array_equal(got[1], want[1])
