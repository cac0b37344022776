"""A landmark that moves in many attributes at once (Algorithm 1 step 2 on correlated points): from
16 on the minima over the points left are taken by warps on their own; the partition equals the
oracle's on both sides of that, with lists in shared and in global memory."""
import numpy as np
import pytest

import oracle
from paper_1412_1947_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,still", [(15, 0), (16, 0), (17, 0), (20, 5), (33, 0), (35, 3), (100, 0), (130, 1)])
@pytest.mark.parametrize("n,N,cap", [(6007, 400, 304), (33, 10, 304), (36000, 5003, 8)])
def test_partition_of_correlated_points(n, N, cap, d, still):
    # every attribute but the `still` constant ones grows along the points
    r = np.random.default_rng(n + d)
    raw = (np.arange(n, dtype=np.float32)[:, None] + 0.25 * r.random((n, d), dtype=np.float32))[r.permutation(n)]
    raw[:, :still] = 2.5
    with B.Job(raw) as job:
        job.option(B.PSCL_OPT_PEEL_GRID, cap)
        job.steps(N, 2, 2, 1, 3)
        perm, off = job.partition()
        x = job.scaled()
    operm, ooff, _ = oracle.peel(x, N, select=True)
    np.testing.assert_array_equal(off, ooff)
    np.testing.assert_array_equal(perm, operm)
