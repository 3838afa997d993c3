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
