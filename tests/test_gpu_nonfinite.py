"""An infinity or a NaN in one pixel of q, k or v reaches the queries whose windows hold it and no other."""
import numpy as np
import pytest
import torch

import oracle
import paper_2304_04237_b200 as sa
from paper_2304_04237_b200 import synth

from test_gpu_fixed_shift import shift_forward
from util import VARIANTS, assert_close, gpu_forward

pytestmark = pytest.mark.gpu

H, W, PIXEL = 13, 37, (6, 17)


def check(forward, k, dtype, sigma_w, what):
    """`forward` of inputs with the pixel's channel 5 of head 1 replaced, against the oracle where the windows do not hold it."""
    x = synth.make_inputs(1, H, W, 2, 32, k, dtype, sigma_w, 0.3, True, seed=40 + k)
    ref = oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], k)
    y, z = np.meshgrid(np.arange(H), np.arange(W), indexing="ij")
    sees = {n: (abs(y - PIXEL[0]) <= k // 2) & (abs(z - PIXEL[1]) <= k // 2) for n in "kv"}
    sees["q"] = (y == PIXEL[0]) & (z == PIXEL[1])
    for name in "qkv":
        for value in (np.inf, -np.inf, np.nan):
            bad = dict(x, **{name: x[name].copy()})
            bad[name][0, PIXEL[0], PIXEL[1], 1, 5] = value
            got = forward(bad)
            other = np.ones(got.shape, bool)
            other[0, :, :, 1][sees[name]] = False
            assert np.isfinite(got[other]).all(), f"{what}: {value} in {name} spreads"
            assert_close(np.where(other, got, ref), ref, dtype, what)
            if np.isnan(value):
                assert np.isnan(got[0, :, :, 1, 5][sees[name]]).all(), f"{what}: {value} in {name} is lost"


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("k", [1, 3, 5, 7, 9])
def test_nonfinite_pixel_fixed_shift(k, dtype):
    check(lambda x: shift_forward(x, k, dtype), k, dtype, 0.0, f"fixed shift k = {k} {dtype}")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("k", [1, 3, 5, 7, 9])
def test_nonfinite_pixel_every_variant(k, dtype):
    ran = 0
    for variant in (None, *VARIANTS.values(), sa.VARIANT_UMMA_SPLIT):
        try:
            check(lambda x: gpu_forward(x, k, dtype, variant), k, dtype, 0.1, f"variant {variant} k = {k} {dtype}")
        except sa.SlideAttnError as e:
            assert e.status == sa.ERR_UNSUPPORTED
            continue
        ran += 1
    assert ran >= 3
