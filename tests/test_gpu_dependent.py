"""Calls that follow one another on a stream and depend on one another: each reads what the one before wrote and overwrites what the one
before read.  Kernels start before the ones ahead of them have finished, so the order rests on what they wait for.  The same calls with
the device idle in between give the bits to compare with.  Shapes: four blocks of pixels and more for a CTA, and a few for the whole chip."""
import pytest
import torch

import paper_2304_04237_b200 as sa

pytestmark = pytest.mark.gpu

SHAPES = [(16, 40, 44, 3), (2, 13, 18, 3)]
BF16, F32 = torch.bfloat16, torch.float32
# (what, window), in turn
CHAINS = [(32, BF16, c) for c in ([("forward", 3)], [("forward", 3), ("forward", 5)], [("forward", 5)], [("forward", 7), ("forward", 3)], [("shift", 3), ("forward", 3)],
                                  [("shift", 7), ("forward", 3)], [("block", 3)], [("block", 3), ("forward", 3)], [("block", 5)], [("train", 3)],
                                  [("train", 3), ("block", 3), ("shift", 3)])] + \
         [(32, F32, c) for c in ([("forward", 3)], [("train", 3), ("forward", 3)], [("shift", 3), ("forward", 3)])] + \
         [(d, t, [("forward", 3)]) for d in (16, 64) for t in (BF16, F32)] + [(16, BF16, [("block", 3)]), (64, BF16, [("block", 3), ("forward", 3)])]


class Step:
    def __init__(self, what, k, shape, d, dtype, gen):
        C, k2 = shape[3] * d, k * k
        self.what = what
        self.ctx = sa.slide_attn_create(*shape, d, k, dtype, False)
        if what == "shift":
            sa.slide_attn_set_fixed_shift(self.ctx, True)
        eye = torch.eye(k2, device="cuda").expand(C, k2, k2)
        self.w = [(eye + (0 if what == "shift" else 0.1) * torch.randn(C, k2, k2, device="cuda", generator=gen)).contiguous() for _ in range(2)]
        self.proj = torch.randn(4, C, C, device="cuda", generator=gen) / C ** 0.5
        self.sums = [torch.empty_like(w) for w in self.w]

    def run(self, b):
        """From the tensors b[0 .. 2] to b[3], which the next call reads; for training on to b[4 .. 6] with the output as its own gradient."""
        if self.what == "block":
            x, out = (t.view(*t.shape[:3], -1) for t in (b[2], b[3]))
            return sa.slide_attn_block_forward(self.ctx, x, self.proj[:3], self.proj[3], *self.w, None, out)
        sa.slide_attn_forward(self.ctx, *b[:3], *self.w, None, b[3])
        if self.what == "train":
            sa.slide_attn_backward(self.ctx, *b[:3], *self.w, None, b[3], *b[4:7], *self.sums, None)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("d,dtype,chain", CHAINS, ids=lambda c: str(c).replace("torch.", ""))
def test_calls_that_depend_on_one_another(d, dtype, chain, shape):
    gen = torch.Generator(device="cuda").manual_seed(d)
    steps = [Step(what, k, shape, d, dtype, gen) for what, k in chain]
    first = [torch.randn(*shape, d, device="cuda", generator=gen).to(dtype) for _ in range(7)]

    def run(idle):
        ring = [t.clone() for t in first]
        for i in range(8):
            if idle:
                torch.cuda.synchronize()
            # b[3] was the first operand of the call before; it is the third one of the next
            steps[i % len(steps)].run([ring[(i + j) % 4] for j in range(4)] + ring[4:])
        return ring

    try:
        want = run(True)
        assert all(bool(t.isfinite().all()) for t in want)
        assert float(want[2].float().std()) > 1e-3               # what the last call wrote
        for _ in range(10):
            assert all(torch.equal(a, b) for a, b in zip(run(False), want))
        assert all(sa.slide_attn_query_status(s.ctx) == sa.OK for s in steps)
    finally:
        for s in steps:
            sa.slide_attn_destroy(s.ctx)
