"""Unequal-sized subclustering (Algorithm 2): the grouping scores only the landmarks around a
point's projection on their line; the partition equals the oracle's, which scores them all in
float64, at window and table sizes from one landmark to the most there can be."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth
from tests.parity import run_oracle

pytestmark = pytest.mark.gpu


def _check(raw, m):
    with B.Job(raw) as j:
        j.steps_unequal(m, 2, 2, 1, 3)
        perm, off = j.partition()
    o = run_oracle(raw, 0, 2, 2, 1, seed=3, unequal_m=m)
    np.testing.assert_array_equal(perm, o.perm)
    np.testing.assert_array_equal(off, o.seg_off)


@pytest.mark.parametrize("n,d,m", [
    (1025, 2, 1), (1023, 2, 2), (3000, 3, 3),            # one tile and a point; no step, one, two
    (5000, 2, 4096), (4000, 8, 4096), (2000, 64, 4096),  # the most: wide windows; beyond the table
    (3000, 128, 193), (2500, 33, 700), (9000, 1, 257),   # generic widths, one attribute
])
def test_partition_equals_the_oracle(n, d, m):
    _check(synth.mixture(n, d, 7, outlier_frac=0.02, seed=7000 + n + m), m)


@pytest.mark.parametrize("m", [1, 2, 50])
def test_points_on_the_line_and_flat_attributes(m):
    # on the landmarks' line (every midpoint a tie), a flat attribute, and nearly all points equal
    t = np.repeat(np.arange(0, 2 * m + 1, dtype=np.float32) / (2 * m), 40)
    _check(np.ascontiguousarray(np.stack([t, t, np.full_like(t, 0.25), 1 - t], axis=1)), m)
    x = np.full((1500, 4), 0.5, np.float32)
    x[700] += np.float32(1e-7)
    _check(x, m)
