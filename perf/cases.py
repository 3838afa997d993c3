"""The work that users of this library have it do, as cases to time and to compare.

One case is one call (or, for training, one forward and one backward) through the public binding, on the
map sizes of hierarchical vision transformers: 56 x 56 and 28 x 28 stages of a batch of images, 128 x 128
crops of a dense-prediction network, and a 14 x 14 map of one image as the smallest call.

    op      "forward"   slide_attn_forward, general (deformed) weights
            "shift"     slide_attn_forward in fixed-shift mode (one-hot weights)
            "block"     slide_attn_block_forward: projections, attention, output projection
            "train"     slide_attn_forward, then slide_attn_backward of its output's gradient
            "host"      slide_attn_forward_host on page-locked host buffers
    B, H, W, heads, head_dim, ksize, dtype ("f32" / "bf16"), bias (truth value): the context's shape
"""
import math

import torch

import paper_2304_04237_b200 as sa

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
SIGMA_W = 0.05          # learned part of the merged depthwise weights, beside the one-hot shift kernels
SIGMA_BIAS = 0.02


def _case(name, op, B, H, W, heads, head_dim, ksize, dtype, bias=True):
    return dict(name=name, op=op, B=B, H=H, W=W, heads=heads, head_dim=head_dim, ksize=ksize, dtype=dtype, bias=bias)


def listed():
    return [
        # one small map of one image in fp32: the smallest call, where latency and launches count
        _case("tiny_f32", "forward", 1, 14, 14, 1, 32, 3, "f32", False),
        # inference of the first stage of a classification backbone, a batch of 64 images
        _case("stage1_bf16", "forward", 64, 56, 56, 2, 32, 3, "bf16"),
        # a later stage on pictures that are not square: more heads, rows that no tile width divides
        _case("ragged_bf16", "forward", 32, 28, 42, 6, 32, 3, "bf16"),
        # a dense-prediction crop at full precision, two images
        _case("crop_f32", "forward", 2, 128, 128, 3, 32, 3, "f32", False),
        # heads twice as wide, as backbones with 64 channels per head have them
        _case("heads64_bf16", "forward", 32, 28, 28, 3, 64, 3, "bf16"),
        # wider windows, the setting of the neighbourhood-size comparison: 5 x 5 on a whole batch ...
        _case("stage1_k5_bf16", "forward", 64, 56, 56, 3, 32, 5, "bf16"),
        # ... and 7 x 7 on a crop
        _case("crop_k7_bf16", "forward", 2, 128, 128, 3, 32, 7, "bf16"),
        # the method without the deformed shifting module: one-hot kernels, plain local attention
        _case("shift_bf16", "shift", 64, 56, 56, 3, 32, 3, "bf16"),
        # a whole attention block of the first stage
        _case("block_bf16", "block", 64, 56, 56, 2, 32, 3, "bf16"),
        # one training step through the module, mixed precision, a whole batch: the largest call
        _case("train_bf16", "train", 64, 56, 56, 3, 32, 3, "bf16"),
        # the same at full precision on a crop
        _case("train_f32", "train", 2, 128, 128, 3, 32, 3, "f32"),
        # a program whose tensors live on the host: copies in, the forward and the copy out
        _case("host_bf16", "host", 2, 128, 128, 3, 32, 3, "bf16"),
    ]


def _elements(c):
    return c["B"] * c["H"] * c["W"] * c["heads"] * c["head_dim"]


# What the largest listed cases work on: elements of one tensor, and elements times k^4 for general weights.
MOST_ELEMENTS = 64 * 56 * 56 * 96
MOST_TAPS = MOST_ELEMENTS * 5 ** 4


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(["forward", "shift", "block", "train", "host"], [45, 15, 15, 15, 10])[0]
    dtype = "bf16" if op == "block" or rng.random() < 0.65 else "f32"
    head_dim, ksize = 32, 3
    if op == "forward":
        if rng.random() < 0.25:
            head_dim = rng.choice([16, 64])
        elif dtype == "bf16":
            ksize = rng.choice([3, 3, 3, 5, 7, 9])
        else:
            ksize = rng.choice([3, 3, 5])
    elif op == "shift":
        ksize = rng.choice([3, 3, 5, 7, 9])
    H = _log_int(rng, 7, 128)
    W = H if rng.random() < 0.4 else _log_int(rng, 7, 128)
    heads = rng.randint(1, 8 if head_dim <= 32 else 4)
    B = _log_int(rng, 1, 64)
    c = dict(op=op, B=B, H=H, W=W, heads=heads, head_dim=head_dim, ksize=ksize, dtype=dtype, bias=rng.random() < 0.7)
    # no dearer than the largest listed case: fp32 storage, other head widths and training do more per element
    elements = MOST_ELEMENTS / 4 if dtype == "f32" or head_dim != 32 or op == "host" else MOST_ELEMENTS
    taps = MOST_TAPS / 16 if dtype == "f32" or head_dim != 32 else MOST_TAPS
    while c["B"] > 1 and (_elements(c) > elements or (op != "shift" and _elements(c) * ksize ** 4 > taps)):
        c["B"] -= 1
    while c["heads"] > 1 and op != "shift" and _elements(c) * ksize ** 4 > taps:
        c["heads"] -= 1
    return c


class _State:
    """What the user's program keeps: the library's handle and its tensors."""

    def __init__(self, c):
        self.case = c
        self.handle = sa.slide_attn_create(c["B"], c["H"], c["W"], c["heads"], c["head_dim"], c["ksize"],
                                           DTYPES[c["dtype"]], c["bias"])
        if c["op"] == "shift":
            sa.slide_attn_set_fixed_shift(self.handle, True)

    def __del__(self):
        handle, self.handle = getattr(self, "handle", None), None
        if handle is not None:
            torch.cuda.synchronize()
            sa.slide_attn_destroy(handle)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(*shape, std=1.0):
        return torch.randn(*shape, device="cuda", generator=gen) * std

    td = DTYPES[c["dtype"]]
    C, k2 = c["heads"] * c["head_dim"], c["ksize"] ** 2
    shape = (c["B"], c["H"], c["W"], c["heads"], c["head_dim"])
    s = _State(c)
    one_hot = torch.eye(k2, device="cuda").expand(C, k2, k2)
    if c["op"] == "shift":
        s.wk, s.wv = one_hot.contiguous(), one_hot.contiguous()
    else:
        s.wk, s.wv = ((one_hot + normal(C, k2, k2, std=SIGMA_W)).contiguous() for _ in range(2))
    s.bias = normal(c["heads"], k2, std=SIGMA_BIAS) if c["bias"] else None
    if c["op"] == "block":
        s.x = normal(c["B"], c["H"], c["W"], C).to(td)
        s.w_qkv = normal(3, C, C, std=C ** -0.5)
        s.w_o = normal(C, C, std=C ** -0.5)
        s.out = torch.empty_like(s.x)
        return s
    s.q, s.k, s.v = (normal(*shape).to(td) for _ in range(3))
    s.out = torch.empty_like(s.q)
    if c["op"] == "train":
        s.dout = normal(*shape).to(td)
        s.dq, s.dk, s.dv = (torch.empty_like(s.q) for _ in range(3))
        s.dwk, s.dwv = torch.empty_like(s.wk), torch.empty_like(s.wv)
        s.dbias = torch.empty_like(s.bias) if c["bias"] else None
    elif c["op"] == "host":
        for n in ("q", "k", "v", "wk", "wv", "bias", "out"):
            t = getattr(s, n)
            if t is not None:
                setattr(s, n, t.cpu().pin_memory())
    return s


def run(s):
    op = s.case["op"]
    if op == "block":
        sa.slide_attn_block_forward(s.handle, s.x, s.w_qkv, s.w_o, s.wk, s.wv, s.bias, s.out)
        return s.out
    if op == "host":
        sa.slide_attn_forward_host(s.handle, s.q, s.k, s.v, s.wk, s.wv, s.bias, s.out)
        return s.out
    sa.slide_attn_forward(s.handle, s.q, s.k, s.v, s.wk, s.wv, s.bias, s.out)
    if op != "train":
        return s.out
    sa.slide_attn_backward(s.handle, s.q, s.k, s.v, s.wk, s.wv, s.bias, s.dout,
                           s.dq, s.dk, s.dv, s.dwk, s.dwv, s.dbias)
    grads = {"dq": s.dq, "dk": s.dk, "dv": s.dv, "dwk": s.dwk, "dwv": s.dwv}
    if s.dbias is not None:
        grads["dbias"] = s.dbias
    return {"out": s.out, **grads}


def work(case):
    """Tensors in and out once each, and the multiply-adds of the method (two operations each): per element of
    a tensor k^4 for each depthwise contraction and k^2 for each product with the window."""
    c = case
    C, k2 = c["heads"] * c["head_dim"], c["ksize"] ** 2
    n = _elements(c)
    size = 4 if c["dtype"] == "f32" else 2
    weights = 2 * C * k2 * k2 * 4 + (c["heads"] * k2 * 4 if c["bias"] else 0)
    forward = n * 2 * (2 * k2 if c["op"] == "shift" else 2 * k2 * k2 + 2 * k2)
    if c["op"] == "block":
        return {"bytes": 2 * n * size + 4 * C * C * 4 + weights, "flops": forward + n * 2 * 4 * C}
    if c["op"] == "train":
        # forward, then da, dq, dk, dv, dwk, dwv beside the products that they share with it
        return {"bytes": 8 * n * size + 2 * weights, "flops": forward + n * 2 * (6 * k2 * k2 + 6 * k2)}
    return {"bytes": 4 * n * size + weights, "flops": forward}


def tolerance(case):
    """About four times what the library shows against the same formulas in 64 bits, over these inputs."""
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "max": 2e-5}              # seen: 4.4e-7, 4.2e-6
    if case["op"] == "block":
        return {"rel": 2e-2, "max": 2e-1}              # 4.8e-3, 4.6e-2: q, k, v and z are rounded to bf16 between its stages
    if case["op"] == "shift" or case["head_dim"] != 32:
        return {"rel": 7e-3, "max": 1.6e-2}            # 1.7e-3, 3.9e-3: fp32 arithmetic, the result rounded to bf16 once
    return {"rel": 1e-2, "max": 1.2e-1}                # 2.6e-3, 2.9e-2: products and softmax weights in bf16 too
