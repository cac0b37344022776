"""Small sets run all their Lloyd iterations in one launch, and widths between the compiled
ones run padded with zeros (Algorithm 1 step 4, Section I): labels of every iteration,
counts and centers equal the one-launch-pair-per-set form's and the oracle's."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth
from tests.parity import compare, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def _run(raw, N, lk, fk, T, plain):
    with B.Job(raw) as job:
        job.option(B.PSCL_OPT_TRACE_LABELS, 1).option(B.PSCL_OPT_PLAIN_LLOYD, int(plain))
        job.steps(N, lk, fk, T, 7)
        out = [*job.local_centers(), *job.result()]
        if T:
            out.append(job.trace(0, T))
        launches = job.kernel_times()["lloyd_assign"][0]
    return out, launches


@pytest.mark.parametrize("n,d,N,lk,fk,T", [
    (700, 1, 256, 9, 2, 6), (771, 2, 257, 30, 3, 9),          # one row per thread, and several
    (16384, 8, 4096, 12, 4, 5), (16388, 5, 4095, 7, 4, 5),    # the largest sets of 8 attributes
    (8194, 16, 2048, 20, 3, 4), (4099, 12, 1025, 40, 6, 4),   # 2 rows per thread
    (3000, 32, 1000, 33, 5, 4), (3000, 17, 1024, 9, 5, 4),    # one
    (4096, 8, 2048, 6, 3, 5), (3075, 4, 1025, 12, 3, 5), (4100, 2, 2050, 9, 3, 5),  # two rows, four
    (1024, 64, 512, 5, 3, 4), (770, 33, 257, 8, 3, 4),        # one wide row per thread
    (500, 128, 250, 4, 2, 4), (600, 100, 200, 6, 2, 4), (400, 65, 190, 9, 2, 4),
    (600, 3, 20, 20, 1, 3),                                   # every row a center: over at once
    (500, 4, 100, 1, 1, 30),                                  # a fixed point after two iterations
    (900, 6, 90, 8, 3, 1), (900, 6, 90, 8, 3, 0),
])
def test_one_launch_equals_the_plain_form(n, d, N, lk, fk, T):
    raw = synth.mixture(n, d, 6, outlier_frac=0.02, seed=6000 + n + d)
    got, launches = _run(raw, N, lk, fk, T, False)
    ref, plain_launches = _run(raw, N, lk, fk, T, True)
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)
    if T > 3:
        assert launches < plain_launches


@pytest.mark.parametrize("d", [1, 3, 9, 13, 20, 25, 33, 50, 65, 100, 129])
def test_padded_widths_equal_the_oracle(d):
    raw = synth.mixture(3000, d, 5, outlier_frac=0.01, seed=6100 + d)
    g = run_gpu(raw, 1300, 11, 7, 3, seed=5)
    compare(g, run_oracle(raw, 1300, 11, 7, 3, seed=5, gpu=g))


@pytest.mark.parametrize("n,d,k", [(1000, 16, 16), (70001, 8, 5), (5003, 64, 300), (400000, 7, 33)])
def test_noalloc_takes_points_at_any_float_boundary(n, d, k):
    import torch
    r = np.random.default_rng(n)
    x = r.random((n, d), dtype=np.float32)
    c = x[:k].copy()
    out = []
    for off in (0, 1):
        flat = torch.zeros(n * d + 4, device="cuda")
        pts = flat[off:off + n * d].view(n, d)
        pts.copy_(torch.from_numpy(x))
        cen = torch.zeros(k * d + 4, device="cuda")[off:off + k * d].view(k, d)
        cen.copy_(torch.from_numpy(c))
        lab = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        sse = torch.zeros(1, dtype=torch.float64, device="cuda")
        B.pscl_assign_sse_noalloc(pts, cen, lab, sse, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        out.append((lab.cpu().numpy(), float(sse)))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
    d64 = ((x[:500, None, :].astype(np.float64) - c[None].astype(np.float64)) ** 2).sum(2)
    best = d64.min(1)
    assert (d64[np.arange(500), out[0][0][:500]] <= best * (1 + 1e-5) + 1e-12).all()
