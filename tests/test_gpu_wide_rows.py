"""Rows of more than 128 attributes: 128 attributes with zero columns between them have the same
float32 distances bit for bit (a zero column adds RN(0 * 0 + acc) = acc), so labels, centers and
sums equal those of the 128 attributes alone, wherever a row's first whole sector lies."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _spread(x, d, r):
    at = np.sort(r.choice(d, x.shape[1], replace=False))
    y = np.zeros((len(x), d), np.float32)
    y[:, at] = x
    return y, at


def _noalloc(x, c, off):
    import torch
    n, d = x.shape
    flat = torch.zeros(n * d + 8, device="cuda")
    pts = flat[off:off + n * d].view(n, d)
    pts.copy_(torch.from_numpy(x))
    lab = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    sse = torch.zeros(1, dtype=torch.float64, device="cuda")
    B.pscl_assign_sse_noalloc(pts, torch.from_numpy(c).cuda(), lab, sse, torch.cuda.current_stream().cuda_stream)
    return lab.cpu().numpy(), sse.cpu().numpy()


@pytest.mark.parametrize("d,off", [(129, 0), (129, 3), (130, 1), (132, 2), (135, 0), (136, 0), (136, 7), (144, 4), (257, 5)])
@pytest.mark.parametrize("n", [200, 5000])
def test_nearest_center_of_wide_rows(d, off, n):
    r = np.random.default_rng(d * 10 + off)
    x = r.random((n, 128), dtype=np.float32)
    c = x[r.choice(n, 30, replace=False)] + np.float32(0.01)
    y, at = _spread(x, d, r)
    e = np.zeros((30, d), np.float32)
    e[:, at] = c
    want, got = _noalloc(x, c, 0), _noalloc(y, e, off)
    np.testing.assert_array_equal(got[0], want[0])
    np.testing.assert_array_equal(got[1], want[1])


@pytest.mark.parametrize("d", [129, 131, 136, 150, 260])
def test_lloyd_of_wide_rows(d):
    r = np.random.default_rng(d)
    sizes, k = np.array([700, 129, 40, 2500, 1]), np.array([20, 9, 40, 120, 1], np.int32)
    x = r.random((int(sizes.sum()), 128), dtype=np.float32)
    y, at = _spread(x, d, r)
    out = []
    for p in (x, y):
        with B.Batch(p, sizes, k) as b:
            b.option(B.PSCL_OPT_TRACE_LABELS, 1)
            b.run(6, 3, B.PSCL_PREC_FP32)
            out.append(b.result() + (b.trace(),))
    (c, lab, sse, tr), (c2, lab2, sse2, tr2) = out
    np.testing.assert_array_equal(tr2, tr)
    np.testing.assert_array_equal(lab2, lab)
    np.testing.assert_array_equal(c2[:, at], c)
    np.testing.assert_array_equal(sse2, sse)
