"""Peels that run side by side in a server wait at their own grids' barriers, so all their CTAs
must be resident at once: the grids together are no more than the SMs hold of any width's peel, and
served jobs of 128 attributes, whose peel takes most of an SM, equal the jobs alone."""
import ctypes as C

import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth


def test_query_rejects_what_has_no_kernel():
    v = C.c_int32()
    assert B.lib().pscl_peel_ctas_per_sm(0, 16, None) == B.PSCL_EINVAL
    for d in (0, -1, 1025):
        assert B.lib().pscl_peel_ctas_per_sm(0, d, C.byref(v)) == B.PSCL_EINVAL


def test_grid_query_rejects_null():
    v = C.c_int32()
    assert B.lib().pscl_server_peel_grid(None, C.byref(v), C.byref(v)) == B.PSCL_EINVAL


@pytest.mark.gpu
def test_side_by_side_peels_of_any_widths_fit_the_device():
    import torch
    per_sm = [B.pscl_peel_ctas_per_sm(d) for d in (1, 2, 3, 4, 7, 8, 16, 32, 33, 64, 100, 128, 129, 1024)]
    assert min(per_sm) >= 1
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with B.Server(slots=1) as srv:
        ctas, side_by_side = B.pscl_server_peel_grid(srv.h)
    assert ctas >= 1 and side_by_side > 1
    assert side_by_side * ctas <= sms * min(per_sm)


@pytest.mark.gpu
def test_side_by_side_peels_of_the_widest_rows():
    # four slots, so four peels at a time: of 128 attributes all, then mixed with narrower ones
    shapes = [(30000, 128, 500, 6, 10), (20011, 128, 400, 6, 8), (41000, 128, 700, 8, 12), (16000, 128, 250, 5, 9),
              (30000, 128, 600, 6, 7), (50000, 64, 900, 8, 20), (25000, 100, 500, 6, 6), (22000, 128, 300, 6, 11)]
    pts = [synth.mixture(n, d, 10, seed=8800 + i) for i, (n, d, *_) in enumerate(shapes)]
    with B.Server(slots=4) as srv:
        tickets = [srv.submit(p, N, lk, fk, 4, 31 + i, B.PSCL_PREC_TC, want_labels=True)
                   for i, (p, (n, d, N, lk, fk)) in enumerate(zip(pts, shapes))]
        got = []
        for t in tickets:
            srv.wait(t, 60_000_000)
            got.append(srv.fetch(t))
    for i, (p, (n, d, N, lk, fk)) in enumerate(zip(pts, shapes)):
        with B.Job(p) as job:
            job.run(N, lk, fk, 4, 31 + i, B.PSCL_PREC_TC)
            c, lab, sse = job.result()
        np.testing.assert_array_equal(got[i][0], c)
        np.testing.assert_array_equal(got[i][1], lab)
        assert got[i][2] == sse
