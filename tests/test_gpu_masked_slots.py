"""A bias of -inf masks a slot: its weight is exactly 0 and the others are those of a softmax without it.  Whole groups of slots
are masked (the first sixteen, everything around the 3 x 3 centre, the first window columns, all but one), so that a softmax
which goes over the slots in parts meets parts without any finite logit."""
import zlib

import numpy as np
import pytest

import oracle
import paper_2304_04237_b200 as sa
from paper_2304_04237_b200 import synth

from test_gpu_fixed_shift import shift_forward
from util import VARIANTS, assert_close, gpu_forward

pytestmark = pytest.mark.gpu


def masks(k):
    k2, r = k * k, k // 2
    s = np.arange(k2)
    centre = (abs(s // k - r) <= 1) & (abs(s % k - r) <= 1)
    out = {"first columns": s % k <= r, "all but the last": s < k2 - 1, "all but the first": s > 0}
    if k > 3:
        out.update({"first sixteen": s < 16, "around the centre": ~centre})
    return out


def masked(shape, k, dtype, mask, sigma_w):
    B, H, W, heads, d = shape
    x = synth.make_inputs(B, H, W, heads, d, k, dtype, sigma_w, 0.3, True, seed=zlib.crc32(repr((shape, k, mask.sum())).encode()) & 0xFFFFFF)
    x["bias"] = np.where(mask, np.float32(-np.inf), x["bias"]).astype(np.float32)
    return x, oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], k)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("k", [3, 5, 7, 9])
def test_masked_slots_every_variant(k, dtype):
    shape = (1, 9, 11, 2, 32)
    ran = 0
    for name, mask in masks(k).items():
        x, ref = masked(shape, k, dtype, mask, 0.1)
        for variant in (None, *VARIANTS.values(), sa.VARIANT_UMMA_SPLIT):
            try:
                got = gpu_forward(x, k, dtype, variant)
            except sa.SlideAttnError as e:
                assert e.status == sa.ERR_UNSUPPORTED
                continue
            assert_close(got, ref, dtype, f"{name}, variant {variant}")
            ran += 1
    assert ran >= 3 * len(masks(k))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("k", [3, 5, 7, 9])
def test_masked_slots_fixed_shift(k, dtype):
    for name, mask in masks(k).items():
        x, ref = masked((1, 9, 37, 2, 32), k, dtype, mask, 0.0)
        assert_close(shift_forward(x, k, dtype), ref, dtype, name)
