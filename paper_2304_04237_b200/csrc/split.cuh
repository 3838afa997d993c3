// Exact splits for the tensor-core kernels that keep fp32 arithmetic: an fp32 value is the sum of three
// bf16 values (its 24 significant bits cut into 8 + 8 + 8 by truncation, so nothing is lost), and the product
// of two bf16 values, which has 16 significant bits, is the sum of two.  A product of two split numbers is then
// a handful of bf16 tensor-core products with fp32 accumulation; the pairs whose factors are both small (below
// 2^-24 of the product) are left out.
//
// The tensor core rounds towards zero whenever it adds to an accumulator (measured: 1 + 2^-24 stays 1), so
// long sums are cut: accumulators are added to fp32 registers, which round to nearest, every few steps.
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace slide_attn {
namespace split {

// two floats -> their upper halves (truncated bf16) in one register, `a` in the low half
__device__ __forceinline__ uint32_t pack_upper(float a, float b) {
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}
// what truncation to bf16 leaves of x (exact)
__device__ __forceinline__ float rest(float x) { return x - __uint_as_float(__float_as_uint(x) & 0xFFFF0000u); }

// (a0, a1) * (b0, b1), and what truncation to bf16 leaves of a pair, as packed fp32 operations
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 ra, ra, rb;\n\t"
        "mov.b64 {%0, %1}, ra;\n\t}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 rest2(float2 x) {
    const float h0 = __uint_as_float(__float_as_uint(x.x) & 0xFFFF0000u), h1 = __uint_as_float(__float_as_uint(x.y) & 0xFFFF0000u);
    float2 d = x;
    ffma2(d.x, d.y, h0, h1, -1.f, -1.f);
    return d;
}

__device__ __forceinline__ float2 lds_f2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

// hi - neg_lo = x * y exactly, per half of the register (barring underflow of the low part), given nx = -x: a multiply and an
// FMA, no negation in between.
__device__ __forceinline__ void product2n(uint32_t x, uint32_t nx, uint32_t y, uint32_t& hi, uint32_t& neg_lo) {
    const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&x), na = *reinterpret_cast<const __nv_bfloat162*>(&nx),
                         b = *reinterpret_cast<const __nv_bfloat162*>(&y);
    const __nv_bfloat162 h = __hmul2_rn(a, b);
    const __nv_bfloat162 l = __hfma2(na, b, h);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    neg_lo = *reinterpret_cast<const uint32_t*>(&l);
}

// four 8 x 8 matrices of 16-bit elements, transposed: the B fragments of a row-major [K][N] tile.
// lane i holds the address of row i % 8 of matrix i / 8.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr) : "memory");
}

}  // namespace split
}  // namespace slide_attn
