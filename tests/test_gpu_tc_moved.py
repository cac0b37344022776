"""The sums of the later Lloyd iterations on the tensor-core path, formed from the rows that
changed their center: counts, centers and every iteration's labels equal the float32 path's,
which adds every row again (Section I's update step)."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,N,lk,fk,T", [
    (1000, 16, 1000, 2, 2, 2),         # one later iteration, one set
    (4227, 16, 129, 5, 40, 9),         # sets one row past a warp's share of 128
    (6001, 32, 511, 256, 17, 6),       # many centers per set: some lose all their members
    (5000, 64, 1283, 100, 256, 7),     # one lane per two attributes, ragged last share
    (300, 16, 20, 20, 3, 5),           # as many centers as rows: nothing moves after the first
])
def test_moved_rows_give_the_same_sums(n, d, N, lk, fk, T):
    raw = synth.mixture(n, d, 12, outlier_frac=0.02, seed=3000 + n + d)
    got = {}
    for name, prec in (("ref", B.PSCL_PREC_FP32), ("tc", B.PSCL_PREC_TC)):
        with B.Job(raw) as job:
            job.option(B.PSCL_OPT_TRACE_LABELS, 1)
            for seed in (5, 6):                  # the second run starts from the first one's buffers
                job.run(N, lk, fk, T, seed, prec)
                c, keff, cnt = job.local_centers()
                fc, lab, sse = job.result()
                got.setdefault(name, []).append((c, keff, cnt, fc, lab, sse, job.trace(0, T), job.trace(1, T)))
    for a, b in zip(got["ref"], got["tc"]):
        for u, v in zip(a, b):
            np.testing.assert_array_equal(u, v)
