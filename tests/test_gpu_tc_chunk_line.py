"""Pooled sets of 128 attributes and more centers than one chunk of the tensor-core search holds: on
both sides of the line from which the chunks serve them, centers, labels and the sum equal the
float32 mode's bit for bit."""
import numpy as np
import pytest

from paper_1412_1947_gb300 import binding as B
from paper_1412_1947_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("local_k", [200, 2559, 2560])       # 8 sets: 1600, 20472 and 20480 pooled rows
@pytest.mark.parametrize("final_k", [128, 129, 300, 800])
def test_pooled_set_equals_float32(local_k, final_k):
    x = synth.mixture(24000, 128, 40, seed=61)
    out = []
    for prec in (B.PSCL_PREC_FP32, B.PSCL_PREC_TC, B.PSCL_PREC_BF16):
        with B.Job(x) as job:
            job.run(3000, local_k, final_k, 2, 9, prec)
            out.append(job.result())
    for c, lab, sse in out[1:]:
        np.testing.assert_array_equal(c, out[0][0])
        np.testing.assert_array_equal(lab, out[0][1])
        assert sse == out[0][2]
