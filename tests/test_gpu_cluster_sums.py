"""The no-allocation SSE of 257 .. 2048 rows is one cluster whose blocks hand their sums to the
first one's shared memory: the shortest-lived blocks (a row tile each, one center), launched back
to back, lose none of them.  The coordinates are small integers and the center 0, so every sum is
exact."""
import pytest

from paper_1412_1947_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [257, 512, 513, 1025, 1800, 2048])
@pytest.mark.parametrize("d,k", [(1, 1), (129, 1), (33, 24)])
def test_no_block_sum_is_lost(n, d, k):
    import torch
    reps = 300
    g = torch.Generator(device="cuda").manual_seed(n * 131 + d)
    x = torch.randint(0, 8, (n, d), generator=g, device="cuda").float()
    c = torch.zeros((k, d), device="cuda")
    lab = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    sse = torch.full((reps,), -1.0, dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    for r in range(reps):
        B.pscl_assign_sse_noalloc(x, c, lab, sse[r:], st)
    torch.cuda.synchronize()
    want = int((x.double() ** 2).sum())
    assert sse.cpu().tolist() == [float(want)] * reps
    assert not lab.any()
