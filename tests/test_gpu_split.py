"""GPU parity of the UMMA_SPLIT variant (fp32 arithmetic on tcgen05 through exact splits) against the oracle.

Tolerances.  fp32: a logit is 36 - 108 tensor-core accumulations, each truncated to 2^-23 of the running sum, and the
softmax and the value sums add a few 2^-23 more: 1e-5 of max(1, |ref|) leaves a factor of about three.  bf16: the same
before one rounding to 8 significant bits (half an ulp: at most 2^-8 of the value)."""
import zlib

import numpy as np
import pytest
import torch

import oracle
import paper_2304_04237_b200 as sa
from paper_2304_04237_b200 import synth

from util import gpu_forward, to_device

pytestmark = pytest.mark.gpu

TIGHT = {"f32": 1e-5, "bf16": 2.0 ** -8 + 1e-5}
# one strip of 4 x 8 pixels, its edges, part of a block, several blocks per team, every head count of a grid
SHAPES = [(1, 1, 1, 1), (1, 4, 8, 1), (2, 5, 9, 2), (1, 2, 2, 3), (1, 14, 14, 1), (2, 17, 13, 3), (1, 33, 47, 2), (3, 28, 42, 6), (19, 28, 28, 8)]


def inputs(shape, d, dtype, sigma_w, bias=True):
    B, H, W, heads = shape
    return synth.make_inputs(B, H, W, heads, d, 3, dtype, sigma_w, 0.3, bias, seed=zlib.crc32(repr((shape, d)).encode()) & 0xFFFFFF)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [16, 32, 64])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_split_variant_matches_oracle(shape, d, dtype):
    for sigma_w, bias in ((0.05, True), (0.4, False)):
        x = inputs(shape, d, dtype, sigma_w, bias)
        ref = oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], 3)
        got = gpu_forward(x, 3, dtype, sa.VARIANT_UMMA_SPLIT)
        err = np.abs(got - ref) / np.maximum(1.0, np.abs(ref))
        assert np.isfinite(got).all() and err.max() <= TIGHT[dtype], (sigma_w, float(err.max()))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [16, 32, 64])
@pytest.mark.parametrize("launches,shape", [(1, (1, 9, 10, 2)), (1, (7, 33, 40, 1)), (2, (18, 31, 40, 3))], ids=["part", "one", "more"])
def test_split_variant_weights_laid_out_by_either_kernel(launches, shape, d, dtype):
    """At most one block per team: the fused kernel lays the weights out, whatever else is in their place later; more: a launch in front
    does, as it does under kernel timing.  Both write the same bytes."""
    x = inputs(shape, d, dtype, 0.05)
    dev = to_device(x, dtype)
    outs = [torch.full_like(dev["q"], float("nan")) for _ in range(2)]
    ctx = sa.slide_attn_create(*shape, d, 3, dev["q"].dtype, True)
    try:
        sa.slide_attn_set_variant(ctx, sa.VARIANT_UMMA_SPLIT)
        assert sa.slide_attn_launches_per_forward(ctx) == launches
        for i, out in enumerate(outs):
            if i:
                sa.slide_attn_profile_begin(ctx)
            sa.slide_attn_forward(ctx, dev["q"], dev["k"], dev["v"], dev["wk"], dev["wv"], dev["bias"], out)
        assert sa.slide_attn_profile_end(ctx)[2] == 1
        assert sa.slide_attn_query_status(ctx) == sa.OK
    finally:
        sa.slide_attn_destroy(ctx)
    assert torch.equal(*outs) and bool(torch.isfinite(outs[0]).all())


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_split_variant_weights_of_any_scale(dtype):
    """Channels whose value weights differ by 2^40."""
    x = inputs((1, 9, 10, 2), 32, dtype, 0.4)
    scale = np.exp2(np.arange(64) % 41 - 20).astype(np.float32)
    x["wv"] = x["wv"] * scale[:, None, None]
    ref = oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], 3)
    got = gpu_forward(x, 3, dtype, sa.VARIANT_UMMA_SPLIT)
    s = scale.reshape(2, 32)
    err = np.abs(got - ref) / s / np.maximum(1.0, np.abs(ref) / s)
    assert err.max() <= TIGHT[dtype], float(err.max())


@pytest.mark.parametrize("power", [-100, 110, 120])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [16, 32, 64])
def test_split_variant_values_of_any_scale(d, dtype, power):
    """Values near both ends of the type's range; the result scales with them exactly."""
    x = inputs((1, 9, 10, 2), d, dtype, 0.4)
    plain = gpu_forward(x, 3, dtype, sa.VARIANT_UMMA_SPLIT)
    x["v"] = x["v"] * np.float32(2.0 ** power)
    assert np.array_equal(gpu_forward(x, 3, dtype, sa.VARIANT_UMMA_SPLIT), plain * 2.0 ** power)


@pytest.mark.parametrize("power", [-60, 60, 112, 118])
@pytest.mark.parametrize("d", [16, 32, 64])
def test_split_variant_products_of_any_scale(d, power):
    """Products q k up to 2^118 times the usual ones, weights as much smaller (from 2^112 on products are cut otherwise; lower parts
    of weights fall below the smallest normal bf16 there, 2^-126: 2^-10 of a product)."""
    x = inputs((1, 9, 10, 2), d, "f32", 0.4)
    ref = oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], 3)
    x["q"] = x["q"] * np.float32(2.0 ** (power // 2))
    x["k"] = x["k"] * np.float32(2.0 ** (power - power // 2))
    x["wk"] = x["wk"] * np.float32(2.0 ** -power)
    got = gpu_forward(x, 3, "f32", sa.VARIANT_UMMA_SPLIT)
    err = (np.abs(got - ref) / np.maximum(1.0, np.abs(ref))).max()
    assert err <= (1e-5 if power < 112 else 2e-3), float(err)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_split_variant_is_repeatable(dtype):
    x = inputs((5, 30, 33, 3), 64, dtype, 0.05)
    a, b = (gpu_forward(x, 3, dtype, sa.VARIANT_UMMA_SPLIT) for _ in range(2))
    assert np.array_equal(a, b)


def test_split_variant_many_calls_same_bits():
    """Four planes a head through a ring of four slots: a slot handed back to TMA before its loads were done lost pixels of a
    plane in one call of about a hundred."""
    gen = torch.Generator(device="cuda").manual_seed(11)
    q, k, v = (torch.randn(19, 28, 28, 8, 64, device="cuda", generator=gen) for _ in range(3))
    wk, wv = (torch.randn(512, 9, 9, device="cuda", generator=gen) * 0.05 for _ in range(2))
    ctx = sa.slide_attn_create(19, 28, 28, 8, 64, 3, torch.float32, False)
    try:
        sa.slide_attn_set_variant(ctx, sa.VARIANT_UMMA_SPLIT)
        want, got = torch.empty_like(q), torch.empty_like(q)
        sa.slide_attn_forward(ctx, q, k, v, wk, wv, None, want)
        wrong = torch.zeros((), dtype=torch.int64, device="cuda")
        for _ in range(1500):
            sa.slide_attn_forward(ctx, q, k, v, wk, wv, None, got)
            wrong += (got != want).any()
        assert int(wrong) == 0 and sa.slide_attn_query_status(ctx) == sa.OK
    finally:
        sa.slide_attn_destroy(ctx)
