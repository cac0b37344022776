"""The peel's fitted key digits and its landmark minima over the points left (Algorithm 1 steps
2-5): the partition equals the oracle's where the digits' range degenerates (equal keys, keys
over many octaves), for widths on both sides of the by-attribute copy's limits and of its
32 x 32 tiles, and where every attribute of the landmark moves at once."""
import numpy as np
import pytest

import oracle
from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth

pytestmark = pytest.mark.gpu


def _points(kind, n, d, seed):
    r = np.random.default_rng(seed)
    if kind == "equal":                    # every key is the same
        return np.full((n, d), 3.0, np.float32)
    if kind == "octaves":                  # keys over sixty octaves, many of them tiny
        return np.exp2(-r.uniform(0, 30, size=(n, d))).astype(np.float32)
    if kind == "levels":                   # three levels per attribute: ties, many holders
        return r.integers(0, 3, size=(n, d)).astype(np.float32)
    if kind == "chain":                    # each round's points hold every minimum
        return (np.arange(n, dtype=np.float32)[:, None] + 0.25 * r.random((n, d), dtype=np.float32))
    return synth.mixture(n, d, 9, outlier_frac=0.02, seed=seed)


@pytest.mark.parametrize("kind,n,d,N", [
    ("equal", 3000, 5, 100), ("equal", 70000, 4, 3000),
    ("octaves", 9001, 1, 150), ("octaves", 40000, 33, 900), ("octaves", 300001, 2, 2000),
    ("levels", 20000, 6, 333), ("levels", 9000, 128, 500),
    ("chain", 5000, 7, 40), ("chain", 6000, 40, 31),
    ("mixture", 8191, 32, 200), ("mixture", 8193, 32, 200),       # in the launch, and before it
    ("mixture", 31, 4, 5), ("mixture", 33, 3, 1), ("mixture", 1300000, 4, 20000),
])
def test_partition_equals_the_oracle(kind, n, d, N):
    with B.Job(_points(kind, n, d, 5000 + n + d)) as job:
        job.steps(N, 2, 2, 1, 3)
        perm, off = job.partition()
        x = job.scaled()
    operm, ooff, _ = oracle.peel(x, N, select=True)
    np.testing.assert_array_equal(off, ooff)
    np.testing.assert_array_equal(perm, operm)
