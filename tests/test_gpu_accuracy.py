"""Where tensor cores stand in for fp32 FMAs the result is no further from 64-bit arithmetic than fp32 FMAs are.

Error: 2-norm of the difference over 2-norm of the oracle's.  Forward: against the STRIP variant (fp32 FMAs, no re-association).  Backward:
against what kernels of fp32 FMAs showed on these very inputs (their sums, unlike these kernels', in one fp32 register per lane)."""
import numpy as np
import pytest

import oracle
import paper_2304_04237_b200 as sa
from oracle import backward as ob
from paper_2304_04237_b200 import synth

from test_gpu_backward import gpu_backward, inputs
from util import gpu_forward

pytestmark = pytest.mark.gpu


def error(got, ref):
    return float(np.linalg.norm(got - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("d", [16, 32, 64])
@pytest.mark.parametrize("sigma_w,q_scale", [(0.05, 1.0), (0.05, 4.0), (0.4, 1.0)])
def test_forward_is_as_exact_as_fp32_fmas(d, sigma_w, q_scale):
    x = synth.make_inputs(2, 28, 30, 2, d, 3, "f32", sigma_w, 0.3, True, seed=d)
    x["q"] = x["q"] * np.float32(q_scale)
    ref = oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], 3)
    split, fma = (error(gpu_forward(x, 3, "f32", v), ref) for v in (sa.VARIANT_UMMA_SPLIT, sa.VARIANT_STRIP))
    assert split <= fma, (split, fma)


# 2 x 28 x 28 x 3 heads
FMA_ERRORS = {"f32": dict(dq=1.95e-7, dk=1.94e-7, dv=1.47e-7, dwk=2.2e-7, dwv=1.8e-7),
              "bf16": dict(dwk=2.14e-7, dwv=1.78e-7)}


@pytest.mark.parametrize("dtype", sorted(FMA_ERRORS))
def test_backward_is_as_exact_as_fp32_fmas(dtype):
    x, dout = inputs((2, 28, 28, 3, 3), dtype)
    ref = ob.backward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], 3, dout)
    got = gpu_backward(x, dout, 3, dtype)[0]
    off = {n: error(got[n], ref[n]) for n in FMA_ERRORS[dtype]}
    assert all(off[n] <= e for n, e in FMA_ERRORS[dtype].items()), off
