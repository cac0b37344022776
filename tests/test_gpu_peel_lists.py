"""The peel's lists in global memory, with gaps where points left and compactions once a quarter is
gone, and the settling of groups of every size (Algorithm 1 steps 2-5): the partition equals the
oracle's on tied, spread and clustered points, with slices on both sides of the key cache."""
import numpy as np
import pytest

import oracle
from paper_1412_1947_gb300 import binding as B
from tests.test_gpu_peel_digits import _points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,d,N,cap", [
    ("equal", 70000, 4, 3000, 16),                       # slices of 4375; every band entry ties
    ("levels", 80001, 6, 1300, 16), ("levels", 66000, 3, 2500, 16),
    ("octaves", 90000, 33, 2000, 20), ("octaves", 140000, 2, 9000, 16),
    ("chain", 66000, 7, 1500, 16), ("chain", 70001, 16, 3001, 17),
    ("mixture", 65535, 8, 700, 16), ("mixture", 65553, 8, 700, 16),      # the cache just fits, or not
    ("mixture", 100000, 128, 4000, 16), ("mixture", 200000, 5, 60000, 16),
    ("mixture", 70000, 4, 69999, 16), ("mixture", 90000, 64, 45, 16),
    ("levels", 4000, 2, 500, 304), ("levels", 6000, 3, 1500, 304),       # groups of 65 entries and more
    ("levels", 9000, 12, 2000, 304), ("equal", 1400, 2, 70, 304),
    ("mixture", 30000, 20, 700, 304), ("mixture", 30001, 12, 900, 304),  # copies by attribute: odd tiles
    ("chain", 9001, 48, 400, 304),
])
def test_partition_equals_the_oracle(kind, n, d, N, cap):
    with B.Job(_points(kind, n, d, 5500 + n + d)) as job:
        job.option(B.PSCL_OPT_PEEL_GRID, cap)
        job.steps(N, 2, 2, 1, 3)
        perm, off = job.partition()
        x = job.scaled()
    operm, ooff, _ = oracle.peel(x, N, select=True)
    np.testing.assert_array_equal(off, ooff)
    np.testing.assert_array_equal(perm, operm)
