"""pscl_assign_sse_noalloc on the tensor cores (from 20480 rows and 32 centers on, with enough
work): labels and
the sum equal the float32 kernel's bit for bit, which the same call runs when the points do
not start on a 16-byte boundary."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _call(x, c, off):
    import torch
    n, d = x.shape
    flat = torch.zeros(n * d + 4, device="cuda")
    pts = flat[off:off + n * d].view(n, d)
    pts.copy_(torch.from_numpy(x))
    lab = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    sse = torch.full((1,), -1.0, dtype=torch.float64, device="cuda")
    for _ in range(2):                       # the second call starts from the first one's scratch
        B.pscl_assign_sse_noalloc(pts, torch.from_numpy(c).cuda(), lab, sse, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return lab.cpu().numpy(), sse.cpu().numpy()


@pytest.mark.parametrize("n,d,k,kind", [
    (160001, 16, 32, "unit"), (20481, 16, 512, "unit"), (50007, 16, 257, "offset"),
    (80007, 32, 33, "unit"), (33000, 32, 256, "big"), (21000, 32, 400, "tiny"),
    (20480, 64, 64, "unit"), (40001, 64, 300, "unit"), (30000, 64, 512, "offset"), (25000, 64, 255, "equal"),
    (70000, 32, 40, "nan point"), (180000, 16, 40, "nan center"), (41000, 64, 33, "inf"),
])
def test_tensor_core_pass_equals_float32(n, d, k, kind):
    r = np.random.default_rng(n + d + k)
    x = r.random((n, d), dtype=np.float32)
    c = x[r.choice(n, k, replace=False)] + r.normal(0, 0.02, (k, d)).astype(np.float32)
    if kind == "offset":                     # far from the origin
        x, c = x + np.float32(4096.0), c + np.float32(4096.0)
    elif kind == "big":
        x, c = x * np.float32(1e15), c * np.float32(1e15)
    elif kind == "tiny":                     # squares below the smallest normal number
        x, c = x * np.float32(1e-21), c * np.float32(1e-21)
    elif kind == "equal":                    # every center twice: the lower index wins
        c[k // 2:2 * (k // 2)] = c[:k // 2]
    elif kind == "nan point":
        x[::1001, 3] = np.nan
    elif kind == "nan center":
        c[7, 2] = np.nan
    elif kind == "inf":
        x[5::2003, 1] = np.inf
        c[4, 0] = -np.inf
    lab, sse = _call(x, c, 0)
    ref, rsse = _call(x, c, 1)
    np.testing.assert_array_equal(lab, ref)
    np.testing.assert_array_equal(sse, rsse)
