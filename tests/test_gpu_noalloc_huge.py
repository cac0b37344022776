"""pscl_assign_sse_noalloc on the tensor cores with coordinates whose squares leave float32:
labels and the sum equal the float32 kernel's bit for bit, which the same call runs when the
points do not start on a 16-byte boundary."""
import numpy as np
import pytest

from tests.test_gpu_noalloc_tc import _call

pytestmark = pytest.mark.gpu


def _signs(r, n, d, a):
    return np.where(r.random((n, d)) < 0.5, -a, a).astype(np.float32)


@pytest.mark.parametrize("d,k,n", [(16, 32, 160001), (32, 34, 80007), (64, 40, 40003)])
def test_rows_beside_centers_of_infinite_norm(d, k, n):
    # all but two centers at +-2e19 (in opposite pairs, so that their mean stays small): their
    # squared norms overflow; a row is a center and noise
    r = np.random.default_rng(d + k)
    c = _signs(r, k // 2, d, 2e19)
    c = np.concatenate([c, -c])
    c[[3, k - 2]] *= np.float32(1e-3)
    x = c[r.integers(0, k, n)] * (1.0 + 1e-3 * r.normal(size=(n, d))).astype(np.float32)
    lab, sse = _call(x, c, 0)
    ref, rsse = _call(x, c, 1)
    np.testing.assert_array_equal(lab, ref)
    np.testing.assert_array_equal(sse, rsse)
    assert len(np.unique(lab)) == k                # rows of every center


@pytest.mark.parametrize("d,k,n", [(64, 33, 41000), (32, 64, 50021)])
def test_rows_infinitely_far_from_every_center(d, k, n):
    # norms^2 of 2.6e38 are finite, the distances of most rows to all centers are not: center 0
    r = np.random.default_rng(7 * d + k)
    a = (2.6e38 / d) ** 0.5
    c, x = _signs(r, k, d, a), _signs(r, n, d, a)
    x[::3] *= np.float32(0.5)
    lab, sse = _call(x, c, 0)
    ref, rsse = _call(x, c, 1)
    np.testing.assert_array_equal(lab, ref)
    np.testing.assert_array_equal(sse, rsse)


@pytest.mark.parametrize("scale", [1e17, 4e17, 1e18, 3e18])
def test_on_both_sides_of_the_line(scale):
    # ||x|| + ||c|| on both sides of 2^63, the distances finite but for a few at 3e18
    r = np.random.default_rng(91)
    n, d, k = 90001, 32, 40
    c = (r.normal(size=(k, d)) * scale).astype(np.float32)
    x = (c[r.integers(0, k, n)] + 0.7 * scale * r.normal(size=(n, d))).astype(np.float32)
    lab, sse = _call(x, c, 0)
    ref, rsse = _call(x, c, 1)
    np.testing.assert_array_equal(lab, ref)
    np.testing.assert_array_equal(sse, rsse)
