"""128 attributes on the tensor cores: point tiles streamed in boxes of 32 attributes, centers
in chunks of up to 128.  Labels, centers and SSE equal the float32 direct path's bit for bit
(Section I's nearest center; the final stage and the SSE pass included)."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth
from tests.parity import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,prec", [("bf16", B.PSCL_PREC_BF16), ("bf16x3", B.PSCL_PREC_BF16X3),
                                       ("tf32", B.PSCL_PREC_TF32), ("tc", B.PSCL_PREC_TC)])
@pytest.mark.parametrize("n,N,lk,fk,T", [
    (5000, 1250, 17, 17, 3),           # the fewest centers served, N = 32
    (9001, 3000, 64, 40, 3),           # two A buffers, ragged tiles
    (9001, 3000, 65, 129, 3),          # one A buffer (N = 80); a last chunk of one center
    (7000, 3500, 128, 200, 3),         # the widest operand B; two chunks
    (40000, 4000, 20, 128, 2),         # one whole chunk
    (60000, 1000, 9, 530, 2),          # local sets on the float32 kernel, five chunks
])
def test_128_attributes_equal_float32(name, prec, n, N, lk, fk, T):
    raw = synth.mixture(n, 128, 30, outlier_frac=0.01, seed=3100 + n + lk)
    ref = run_gpu(raw, N, lk, fk, T, seed=4)
    got = run_gpu(raw, N, lk, fk, T, seed=4, prec=prec)
    np.testing.assert_array_equal(got.trace_local, ref.trace_local)
    np.testing.assert_array_equal(got.local_centers, ref.local_centers)
    np.testing.assert_array_equal(got.trace_final, ref.trace_final)
    np.testing.assert_array_equal(got.final_centers, ref.final_centers)
    np.testing.assert_array_equal(got.labels, ref.labels)
    assert got.sse == ref.sse
    if lk > 16:                        # the local stage ran on the tensor cores
        assert got.assigned >= n * T
    print(f"{name} n={n} k={lk}: re-scored {got.rechecked} of {got.assigned} rows")
