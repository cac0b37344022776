"""Groups of band entries that tie by the hundred (Algorithm 1 steps 2-5): up to 128 of them are
ranked one by one, up to 1024 sorted, more cut by selection; the partition equals the oracle's on
repeated rows, whose order is the index alone, and on permuted ones, whose float64 distances differ
in the last bits only."""
import numpy as np
import pytest

import oracle
from paper_1412_1947_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _points(kind, copies, groups, d, r):
    base = r.random((groups, d))
    base[0] = 0.0
    rows = np.repeat(base, copies, axis=0)
    if kind == "permuted":
        rows = np.take_along_axis(rows, r.random(rows.shape).argsort(1), 1)
    return rows[r.permutation(len(rows))].astype(np.float32)


@pytest.mark.parametrize("kind,copies,groups,d,N,cap", [
    ("repeated", 127, 60, 1, 900, 304), ("repeated", 129, 60, 3, 901, 304), ("repeated", 200, 50, 2, 330, 304),
    ("repeated", 513, 30, 1, 1000, 304), ("repeated", 1024, 20, 4, 1500, 304), ("repeated", 1025, 20, 1, 1500, 304),
    ("repeated", 2100, 12, 2, 1300, 304), ("repeated", 700, 110, 1, 5001, 16), ("repeated", 300, 250, 5, 2999, 16),
    ("permuted", 128, 60, 8, 700, 304), ("permuted", 150, 60, 8, 701, 304), ("permuted", 600, 20, 16, 1000, 304),
    ("permuted", 1000, 20, 40, 1999, 304), ("permuted", 1100, 20, 8, 1999, 304), ("permuted", 400, 200, 12, 6001, 16),
])
def test_partition_of_tied_groups(kind, copies, groups, d, N, cap):
    raw = _points(kind, copies, groups, d, np.random.default_rng(copies * 31 + d))
    with B.Job(raw) as job:
        job.option(B.PSCL_OPT_PEEL_GRID, cap)
        job.steps(N, 2, 2, 1, 3)
        perm, off = job.partition()
        x = job.scaled()
    operm, ooff, _ = oracle.peel(x, N, select=True)
    np.testing.assert_array_equal(off, ooff)
    np.testing.assert_array_equal(perm, operm)


@pytest.mark.parametrize("n,d,levels,N", [(10251, 3, 4, 926), (30000, 2, 3, 1001), (20000, 16, 2, 777), (5000, 1, 9, 410)])
def test_partition_where_most_points_hold_a_minimum(n, d, levels, N):
    raw = np.random.default_rng(n + d).integers(0, levels, size=(n, d)).astype(np.float32)
    with B.Job(raw) as job:
        job.steps(N, 2, 2, 1, 3)
        perm, off = job.partition()
        x = job.scaled()
    operm, ooff, _ = oracle.peel(x, N, select=True)
    np.testing.assert_array_equal(off, ooff)
    np.testing.assert_array_equal(perm, operm)
