"""Calls recorded in a CUDA graph (after a first call, which may allocate) replay with new inputs, and two contexts on two streams do not
disturb each other: the kernels of a call are chained by programmatic launches, which both have to keep in order."""
import pytest
import torch

import paper_2304_04237_b200 as sa

pytestmark = pytest.mark.gpu

FORWARDS = [(32, 3, torch.bfloat16), (32, 3, torch.float32), (16, 3, torch.bfloat16), (64, 3, torch.float32), (32, 5, torch.bfloat16), (32, 7, torch.bfloat16),
            (32, 1, torch.bfloat16), (32, 5, torch.float32), (24, 3, torch.float32)]


class Call:
    """A forward (fixed shift or not), a forward and backward, or a block with tensors of its own."""

    def __init__(self, op, d, k, dtype, seed):
        B, H, W, heads = 2, 21, 27, 3
        gen = torch.Generator(device="cuda").manual_seed(seed)
        self.op, C, k2 = op, heads * d, k * k
        self.ctx = sa.slide_attn_create(B, H, W, heads, d, k, dtype, False)
        if op == "shift":
            sa.slide_attn_set_fixed_shift(self.ctx, True)
        n = {"block": 1, "train": 4}.get(op, 3)
        self.maps = [torch.empty(B, H, W, heads, d, device="cuda", dtype=dtype) for _ in range(n)]
        eye = torch.eye(k2, device="cuda").expand(C, k2, k2)
        self.w = [(eye + (0 if op == "shift" else 0.1) * torch.randn(C, k2, k2, device="cuda", generator=gen)).contiguous() for _ in range(2)]
        self.proj = [torch.randn(m, C, C, device="cuda", generator=gen) / C ** 0.5 for m in (3, 1)]
        self.outs = [torch.empty_like(self.maps[0]) for _ in range(4 if op == "train" else 1)]
        self.sums = [torch.empty_like(w) for w in self.w]
        self.fill(seed)

    def fill(self, seed):
        gen = torch.Generator(device="cuda").manual_seed(seed + 1000)
        for m in self.maps:
            m.copy_(torch.randn(m.shape, device="cuda", generator=gen))

    def run(self):
        if self.op == "block":
            x, out = (t.view(*t.shape[:3], -1) for t in (self.maps[0], self.outs[0]))
            return sa.slide_attn_block_forward(self.ctx, x, self.proj[0], self.proj[1][0], *self.w, None, out)
        sa.slide_attn_forward(self.ctx, *self.maps[:3], *self.w, None, self.outs[0])
        if self.op == "train":
            sa.slide_attn_backward(self.ctx, *self.maps[:3], *self.w, None, self.maps[3], *self.outs[1:], *self.sums, None)

    def result(self):
        torch.cuda.synchronize()
        assert sa.slide_attn_query_status(self.ctx) == sa.OK
        return [t.clone() for t in self.outs]


CALLS = [("forward", *f) for f in FORWARDS] + [("shift", 32, k, t) for k in (3, 7) for t in (torch.bfloat16, torch.float32)] + \
    [("train", 32, 3, torch.bfloat16), ("train", 32, 3, torch.float32), ("train", 32, 1, torch.float32), ("block", 32, 3, torch.bfloat16), ("block", 16, 3, torch.bfloat16)]


@pytest.mark.parametrize("call", CALLS, ids=lambda c: "-".join(map(str, c)))
def test_capture_and_replay(call):
    c = Call(*call, seed=1)
    try:
        c.run()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            c.run()
            c.run()
        for seed in (2, 3):
            c.fill(seed)
            for t in c.outs:
                t.fill_(float("nan"))
            graph.replay()
            got = c.result()
            c.run()
            assert all(torch.equal(a, b) for a, b in zip(got, c.result()))
        del graph
    finally:
        sa.slide_attn_destroy(c.ctx)


@pytest.mark.parametrize("call", CALLS, ids=lambda c: "-".join(map(str, c)))
def test_two_contexts_on_two_streams(call):
    a, b = Call(*call, seed=4), Call(*call, seed=5)
    try:
        want = []
        for c in (a, b):
            c.run()
            want.append(c.result())
        streams = [torch.cuda.Stream() for _ in range(2)]
        for _ in range(25):
            for c, s in zip((a, b), streams):
                with torch.cuda.stream(s):
                    c.run()
        for c, w in zip((a, b), want):
            assert all(torch.equal(x, y) for x, y in zip(c.result(), w))
    finally:
        sa.slide_attn_destroy(a.ctx)
        sa.slide_attn_destroy(b.ctx)
