"""Served jobs whose peels run side by side, some sharing the device and one that runs alone
(more than 2^20 points): every result equals the job's own."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth

pytestmark = pytest.mark.gpu


def test_side_by_side_peels_equal_the_jobs_alone():
    shapes = [(20000, 32, 400, 8, 12), (60000, 8, 1000, 8, 20), ((1 << 20) + 77, 4, 30000, 8, 16),
              (30000, 16, 600, 20, 9), (9000, 5, 200, 6, 5), (50000, 32, 900, 9, 30)]
    pts = [synth.mixture(n, d, 10, seed=7500 + i) for i, (n, d, *_) in enumerate(shapes)]
    with B.Server(slots=5) as srv:
        tickets = [srv.submit(p, N, lk, fk, 4, 11 + i, B.PSCL_PREC_TC, want_labels=True)
                   for i, (p, (n, d, N, lk, fk)) in enumerate(zip(pts, shapes))]
        got = []
        for t in tickets:
            srv.wait(t, 60_000_000)
            got.append(srv.fetch(t))
    for i, (p, (n, d, N, lk, fk)) in enumerate(zip(pts, shapes)):
        with B.Job(p) as job:
            job.run(N, lk, fk, 4, 11 + i, B.PSCL_PREC_TC)
            c, lab, sse = job.result()
        np.testing.assert_array_equal(got[i][0], c)
        np.testing.assert_array_equal(got[i][1], lab)
        assert got[i][2] == sse
