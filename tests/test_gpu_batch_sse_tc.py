"""A batch's labels and per-instance SSE from the tensor-core pass (large batches in a
tensor-core mode) equal the float32 pass's bit for bit."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,prec", [("tc", B.PSCL_PREC_TC), ("bf16", B.PSCL_PREC_BF16)])
@pytest.mark.parametrize("d,count,kmax", [(16, 12, 40), (32, 9, 256), (64, 8, 70), (128, 8, 90)])
def test_batch_sse_equals_float32(name, prec, d, count, kmax):
    r = np.random.default_rng(8100 + d)
    sizes = np.concatenate([[1, 1025, 300], r.integers(10000, 40000, size=count)]).astype(np.int64)
    sizes[-1] += max(0, 164000 - int(sizes.sum()))      # enough rows for the tensor-core pass
    k = r.integers(2, kmax + 1, size=len(sizes)).astype(np.int32)
    k[4] = kmax
    raw = np.concatenate([synth.mixture(int(m), d, max(2, int(q) // 2), seed=8200 + i)
                          for i, (m, q) in enumerate(zip(sizes, k))])
    out = []
    for p in (B.PSCL_PREC_FP32, prec):
        with B.Batch(raw, sizes, k) as b:
            b.run(3, 5, p)
            out.append(b.result())
    for u, v in zip(*out):
        np.testing.assert_array_equal(u, v)
