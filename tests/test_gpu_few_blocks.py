"""The no-allocation SSE (Eq. 1): up to 2048 rows are one cluster of blocks, more take a ticket; labels
equal each other's and the sum float64's within the float32 distances' error."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,k", [(1, 1), (16, 16), (5, 700), (64, 30), (129, 9)])
def test_noalloc_on_both_sides_of_a_cluster(d, k):
    # a set of up to 2048 rows takes the cluster; the same rows twice over, past it, the ticket
    import torch
    r = np.random.default_rng(d + k)
    x = torch.from_numpy(r.random((2049, d), dtype=np.float32)).cuda()
    c = torch.from_numpy(r.random((k, d), dtype=np.float32)).cuda()
    c64, x64 = c.double().cpu().numpy(), x.double().cpu().numpy()
    st = torch.cuda.current_stream().cuda_stream
    for n in (1, 255, 256, 257, 1000, 2047, 2048, 2049):
        lab = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        big = torch.full((n + 4098,), -1, dtype=torch.int32, device="cuda")
        sse, sse2 = torch.full((1,), -1.0, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
        B.pscl_assign_sse_noalloc(x[:n], c, lab, sse, st)
        B.pscl_assign_sse_noalloc(torch.cat([x[:n], x, x]).contiguous(), c, big, sse2, st)
        torch.cuda.synchronize()
        got = lab.cpu().numpy()
        np.testing.assert_array_equal(got, big.cpu().numpy()[:n])
        # the sum of the float32 distances of these labels, each within (d + 2) 2^-23 of float64's
        want = ((x64[:n] - c64[got]) ** 2).sum()
        assert abs(float(sse) - want) <= (d + 4) * 2.0 ** -23 * want + 1e-30

