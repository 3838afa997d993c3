"""GPU parity of the MMA_WIDE variant where its schedule can go wrong: one tile and its edges, an odd tile (the second tile of
a block missing), teams without a block in the last round (k >= 7 streams the weights for both teams), several rounds of the
weight ring.  Tolerance as for every bf16 variant (products and softmax weights rounded to bf16)."""
import zlib

import numpy as np
import pytest

import oracle
import paper_2304_04237_b200 as sa
from paper_2304_04237_b200 import synth

from util import assert_close, gpu_forward
from oracle.block import round_bf16

pytestmark = pytest.mark.gpu

SHAPES = [(1, 8, 8, 1), (1, 9, 17, 1), (1, 3, 40, 2), (3, 24, 40, 8), (6, 40, 40, 8)]


@pytest.mark.parametrize("k", [3, 5, 7, 9])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_wide_variant_matches_oracle(shape, k):
    B, H, W, heads = shape
    x = synth.make_inputs(B, H, W, heads, 32, k, "bf16", 0.05, 0.3, True, seed=zlib.crc32(repr((shape, k)).encode()) & 0xFFFFFF)
    ref = oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], k)
    a, b = (gpu_forward(x, k, "bf16", sa.VARIANT_MMA_WIDE) for _ in range(2))
    assert_close(a, ref, "bf16", f"{shape} {k}")
    assert np.array_equal(a, b)


@pytest.mark.parametrize("H", [45, 56])
def test_k5_kernel_with_many_blocks_matches_oracle(H):
    """Nine blocks per CTA, eleven for H = 56, more than any of its rings has slots; edges in both directions.  126 tiles, 147: the second
    tile of the last block is missing."""
    x = synth.make_inputs(3, H, 51, 19, 32, 5, "bf16", 0.05, 0.3, False, seed=55)
    ref = oracle.forward(x["q"], x["k"], x["v"], x["wk"], x["wv"], x["bias"], 5)
    a, b = (gpu_forward(x, 5, "bf16", sa.VARIANT_MMA_WIDE) for _ in range(2))
    assert_close(a, ref, "bf16")
    assert np.array_equal(a, b)


def as_documented(x, k):
    """The kernel's arithmetic in 64 bits, rounded where it rounds: products q k, what the weights differ from the one-hot kernels by,
    and on the value side's learned part exp(logit - largest) are bf16; the result is rounded once."""
    B, H, W, heads, d = x["q"].shape
    r, k2 = k // 2, k * k
    out = np.empty(x["q"].shape)
    for h in range(heads):
        q, kk, v = (x[n][:, :, :, h].astype(np.float64) for n in ("q", "k", "v"))
        win = lambda t: np.stack([np.pad(t, ((0, 0), (r, r), (r, r), (0, 0)))[:, y:y + H, z:z + W] for y in range(k) for z in range(k)], 3)
        dk, dv = (round_bf16(x[n][h * d:(h + 1) * d] - np.eye(k2, dtype=np.float32)).astype(np.float64) for n in ("wk", "wv"))
        p = round_bf16((q[:, :, :, None] * win(kk)).astype(np.float32)).astype(np.float64)
        logits = (np.einsum("bhwtc,cst->bhws", p, dk, optimize=True) + p.sum(4)) / d ** 0.5 + (0 if x["bias"] is None else x["bias"][h])
        e = np.exp(logits - logits.max(3, keepdims=True))
        a = np.einsum("bhws,cst->bhwtc", round_bf16(e.astype(np.float32)).astype(np.float64), dv, optimize=True) + e[..., None]
        out[:, :, :, h] = (a * win(v)).sum(3) / e.sum(3)[..., None]
    return round_bf16(out.astype(np.float32)).astype(np.float64)


@pytest.mark.parametrize("k", [5, 7, 9])
def test_wide_variant_rounds_where_it_says(k):
    """What is left beside the documented roundings: fp32 sums (1e-6 of a result: one in a few hundred falls on the other side of a
    rounding, 2^-8 of it: 2-norm about 2e-4) and weights e as two bf16 (2^-17).  Softmax weights rounded after their division give 1.6e-3."""
    x = synth.make_inputs(2, 19, 26, 2, 32, k, "bf16", 0.2, 0.3, True, seed=90 + k)
    want, got = as_documented(x, k), gpu_forward(x, k, "bf16", sa.VARIANT_MMA_WIDE)
    off = float(np.linalg.norm(got - want) / np.linalg.norm(want))
    assert off <= 5e-4, off
