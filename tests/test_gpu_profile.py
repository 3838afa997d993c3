"""Kernel timing: the main kernel's time leaves the weight re-layout out, whichever variant runs."""
import pytest
import torch

import paper_2304_04237_b200 as sa

pytestmark = pytest.mark.gpu


def gap_us(variant, heads, head_dim, k, dtype):
    """Mean of (all kernels) - (main kernel) of a forward."""
    C, k2 = heads * head_dim, k * k
    q = torch.randn(1, 8, 8, heads, head_dim, device="cuda").to(dtype)
    w = torch.randn(C, k2, k2, device="cuda") * 0.05
    out = torch.empty_like(q)
    ctx = sa.slide_attn_create(1, 8, 8, heads, head_dim, k, dtype, False)
    try:
        sa.slide_attn_set_variant(ctx, variant)
        for _ in range(3):
            sa.slide_attn_forward(ctx, q, q, q, w, w, None, out)
        sa.slide_attn_profile_begin(ctx)
        for _ in range(50):
            sa.slide_attn_forward(ctx, q, q, q, w, w, None, out)
            torch.cuda.synchronize()
        forward_ms, main_ms, n = sa.slide_attn_profile_end(ctx)
        assert n == 50
    finally:
        sa.slide_attn_destroy(ctx)
    return (forward_ms - main_ms) * 1e3


@pytest.mark.parametrize("variant,head_dim,k,dtype", [(sa.VARIANT_UMMA_SPLIT, 64, 3, torch.float32), (sa.VARIANT_MMA_WIDE, 32, 5, torch.bfloat16),
                                                      (sa.VARIANT_UMMA_TS, 32, 3, torch.bfloat16), (sa.VARIANT_STRIP, 64, 3, torch.float32)])
def test_main_time_is_without_the_weight_layout(variant, head_dim, k, dtype):
    """A launch of 16 heads' weights takes 3 us and more; DIRECT, which lays nothing out, shows what two events on end take."""
    assert gap_us(variant, 16, head_dim, k, dtype) >= gap_us(sa.VARIANT_DIRECT, 16, head_dim, k, dtype) + 1.5
