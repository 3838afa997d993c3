// Backward pass of the fused forward (training through the module, Sec. 4.3 / Fig. 4 (1); the paper prints no backward
// formulas: these are the derivatives of Eq. 2 with the depthwise convolution of Eq. 12 inside).  head_dim 32, fp32 or bf16
// storage.  The dispatch for k = 3 (bwd_team_kernel.cu, bwd_weight_umma_kernel.cu, bwd_weight_kernel.cu) and the kernel for
// k = 1, where a window is its pixel.  With g = d(loss)/d(out):
//
//   a = softmax over the one slot of scale * sum_c q[c] k[c] wk[c] + bias        da = sum_c g[c] v[c] wv[c]
//   dl = a (da - a da)      dbias = sum over pixels of dl
//   dq[c] = scale * k[c] dl wk[c]      dk[c] = scale * q[c] dl wk[c]      dwk[c] = scale * sum over pixels of dl q[c] k[c]
//   dv[c] = g[c] a wv[c]               dwv[c] = sum over pixels of a g[c] v[c]
//
// (a is 1 and dl 0 unless something is not finite.)  Four lanes a pixel, eight channels each; a CTA has one head and keeps the
// sums of its pixels in registers.
//
// Bound by memory traffic (four tensors in, three out), with one CTA of 512 threads per SM in flight: 64 x 56 x 56, 3 heads, bf16 91 us
// (3.0 TB/s), fp32 145 us (3.7 TB/s); the window kernels, written for any k, that ran this before: 126 and 186 us.  Four CTAs of 256 per SM
// took 77 and 109 us, but four times the additions to global memory, each rounded: error of dwv against 64 bits 2.4e-7 and 2.9e-7, here
// 1.6e-7 and 1.9e-7, before 2.5e-7 and 4.5e-7.
#include "bwd_common.cuh"
#include "ptx.cuh"

namespace slide_attn {

namespace {

constexpr int kHeadDim = 32, kThreads = 512, kPixels = kThreads / 4;       // pixels of a CTA at a time
constexpr int kSums = 2 * kHeadDim + 1;                                    // dwk, dwv, dbias
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ void load8(const float* p, float (&f)[8]) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&f)[8]) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
    f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x); f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
    f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z); f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
}
__device__ __forceinline__ void store8(float* p, const float (&f)[8]) {
    reinterpret_cast<float4*>(p)[0] = make_float4(f[0], f[1], f[2], f[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(f[4], f[5], f[6], f[7]);
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&f)[8]) {
    *reinterpret_cast<uint4*>(p) = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
}

template <typename T>
struct OneParams {
    const T* q;
    const T* k;
    const T* v;
    const T* g;
    const float* wk;
    const float* wv;
    const float* bias;
    T* dq;
    T* dk;
    T* dv;
    float* dwk;
    float* dwv;
    float* dbias;
    long long pixels;
    int heads;
    float scale;
};

template <typename T>
__global__ void __launch_bounds__(kThreads)
bwd_one_kernel(const OneParams<T> P)
{
    __shared__ float s_sum[kThreads / 32][kSums];
    const int h = blockIdx.x % P.heads, rank = blockIdx.x / P.heads, nrank = (int)gridDim.x / P.heads;
    const int lane = threadIdx.x & 31, c0 = 8 * (lane & 3);
    float wk[8], wv[8], dwk[8], dwv[8], dbias = 0.f;
    load8(P.wk + h * kHeadDim + c0, wk);
    load8(P.wv + h * kHeadDim + c0, wv);
#pragma unroll
    for (int c = 0; c < 8; ++c) { dwk[c] = 0.f; dwv[c] = 0.f; }
    const float bias = P.bias ? P.bias[h] * kLog2e : 0.f;
    auto quad_sum = [](float x) {
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        return x + __shfl_xor_sync(0xffffffffu, x, 2);
    };
    for (long long first = (long long)rank * kPixels; first < P.pixels; first += (long long)nrank * kPixels) {
        const long long pix = first + (threadIdx.x >> 2);
        const bool in = pix < P.pixels;
        const size_t at = ((size_t)pix * P.heads + h) * kHeadDim + c0;
        float q[8] = {}, k[8] = {}, v[8] = {}, g[8] = {}, l = 0.f, da = 0.f;
        if (in) { load8(P.q + at, q); load8(P.k + at, k); load8(P.v + at, v); load8(P.g + at, g); }
#pragma unroll
        for (int c = 0; c < 8; ++c) { l = fmaf(q[c] * k[c], wk[c], l); da = fmaf(g[c] * v[c], wv[c], da); }
        l = fmaf(quad_sum(l), P.scale * kLog2e, bias);
        da = quad_sum(da);
        float a = fast_exp2(l - l);
        a *= 1.f / a;
        const float dl = a * (da - a * da);
        float dq[8], dk[8], dv[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            dq[c] = dl * wk[c] * k[c] * P.scale;
            dk[c] = dl * wk[c] * q[c] * P.scale;
            dv[c] = a * wv[c] * g[c];
        }
        if (in) {
#pragma unroll
            for (int c = 0; c < 8; ++c) { dwk[c] = fmaf(dl, q[c] * k[c], dwk[c]); dwv[c] = fmaf(a, g[c] * v[c], dwv[c]); }
            if ((lane & 3) == 0) dbias += dl;
            store8(P.dq + at, dq); store8(P.dk + at, dk); store8(P.dv + at, dv);
        }
    }
    auto column_sum = [](float x) {                              // over the lanes with the same channels
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        return x;
    };
    float* mine = s_sum[threadIdx.x >> 5];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float sk = column_sum(dwk[c]), sv = column_sum(dwv[c]);
        if (lane < 4) { mine[c0 + c] = sk; mine[kHeadDim + c0 + c] = sv; }
    }
    dbias = column_sum(dbias);
    if (lane == 0) mine[2 * kHeadDim] = dbias;
    __syncthreads();
    const int i = threadIdx.x;
    if (i >= kSums) return;
    float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) sum[w & 3] += s_sum[w][i];
    const float x = (sum[0] + sum[1]) + (sum[2] + sum[3]);
    if (i < kHeadDim) atomicAdd(P.dwk + h * kHeadDim + i, x * P.scale);
    else if (i < 2 * kHeadDim) atomicAdd(P.dwv + h * kHeadDim + i - kHeadDim, x);
    else if (P.dbias) atomicAdd(P.dbias + h, x);
}

template <typename T>
cudaError_t launch_one(const Problem& p, const BackwardArgs& ga, int num_sms, cudaStream_t stream) {
    const size_t wbytes = (size_t)p.heads * kHeadDim * sizeof(float);
    cudaError_t e = cudaMemsetAsync(ga.dwk, 0, wbytes, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ga.dwv, 0, wbytes, stream);
    if (e == cudaSuccess && ga.dbias) e = cudaMemsetAsync(ga.dbias, 0, (size_t)p.heads * sizeof(float), stream);
    if (e != cudaSuccess) return e;
    OneParams<T> P;
    P.q = static_cast<const T*>(p.q); P.k = static_cast<const T*>(p.k); P.v = static_cast<const T*>(p.v); P.g = static_cast<const T*>(ga.dout);
    P.wk = p.wk; P.wv = p.wv; P.bias = p.bias;
    P.dq = static_cast<T*>(ga.dq); P.dk = static_cast<T*>(ga.dk); P.dv = static_cast<T*>(ga.dv);
    P.dwk = ga.dwk; P.dwv = ga.dwv; P.dbias = ga.dbias;
    P.pixels = (long long)p.B * p.H * p.W; P.heads = p.heads; P.scale = 1.f / sqrtf((float)kHeadDim);
    const long long all = (P.pixels + kPixels - 1) / kPixels;
    long long per_head = ((long long)num_sms + p.heads - 1) / p.heads;      // few: what they add to global memory is rounded each time
    if (per_head > all) per_head = all;
    bwd_one_kernel<T><<<(unsigned)(per_head * p.heads), kThreads, 0, stream>>>(P);
    return cudaGetLastError();
}

}  // namespace

bool backward_supports(int head_dim, int ksize) {
    return head_dim == kHeadDim && (ksize == 1 || ksize == 3) && tensor_map_available();
}

size_t backward_workspace_bytes(int B, int H, int W, int heads, int ksize, bool compact) {
    return ksize == 3 ? bwd_team_workspace_bytes(B, H, W, heads, compact) : 0;
}

// `ws`: backward_workspace_bytes of scratch.
cudaError_t launch_backward(const Problem& p, const BackwardArgs& ga, void* ws, bool compact, int* d_status, int num_sms, cudaStream_t stream) {
    if (p.ksize == 1)
        return p.dtype == SLIDE_ATTN_BF16 ? launch_one<__nv_bfloat16>(p, ga, num_sms, stream) : launch_one<float>(p, ga, num_sms, stream);
    const BwdScratch s = bwd_scratch(ws, compact, ga.dv, p.B, p.H, p.W, p.heads);
    cudaError_t e = launch_bwd_team(BwdPass::point, p, ga, s, d_status, num_sms, stream);
    if (e != cudaSuccess) return e;
    e = p.dtype == SLIDE_ATTN_BF16 ? launch_bwd_weight_umma(p, ga, s, d_status, num_sms, stream) : launch_bwd_weight_mma(p, ga, s, d_status, num_sms, stream);
    // last of all: it may write over rows that the weight gradients are made of
    return e == cudaSuccess ? launch_bwd_team(BwdPass::gather, p, ga, s, d_status, num_sms, stream) : e;
}

}  // namespace slide_attn
