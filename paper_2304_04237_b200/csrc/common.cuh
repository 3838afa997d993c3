// Shared declarations of the slide-attention library: problem description, element access,
// and the launchers each kernel file exports to the API layer.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "slide_attn.h"

namespace slide_attn {

// One forward problem.  Channel c = h*head_dim + e; C = heads*head_dim; k2 = ksize*ksize.
struct Problem {
    int B, H, W, heads, head_dim, ksize;
    int has_bias;
    slide_attn_dtype dtype;
    const void* q;
    const void* k;
    const void* v;
    const float* wk;     // [C][k2 slot][k2 tap]
    const float* wv;
    const float* bias;   // [heads][k2] or nullptr
    void* out;
};

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_float(float x);
template <> __device__ __forceinline__ float from_float<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_float<__nv_bfloat16>(float x) {
    return __float2bfloat16_rn(x);
}

// TMA tensor map of a [B][H][W][C] tensor (bf16: elem_bytes 2, fp32: 4) seen as 4-D (C, W, H, B) with
// a box of box_c channels x box_w columns x box_h rows; out-of-map elements read as zero.
bool tensor_map_available();
bool make_tile_map(CUtensorMap* map, const void* base, int elem_bytes, int B, int H, int W, int C,
                   int box_c, int box_w, int box_h);

// Launches with programmatic stream serialisation: the kernel may start before the one ahead of it in the stream has finished and
// has to execute griddepcontrol.wait before it touches anything that one may write or read, and in any case before it completes:
// whoever waits for it takes all that was launched earlier as complete.  The prep kernels wait first of all and only then let the
// main kernel behind them start, so a main kernel never runs beside what was ahead of its prep kernel.  Chained so, back-to-back forwards have no launch gap between them.
// Kernels that lay their weights out themselves, and projections that no prep or check kernel follows, let the next one start when their
// last loads are sent for: 2 x 56 x 56, 2 heads, bf16, k = 3 7.3 us -> 6.2, block 4 x 28 x 28, 6 heads 17.6 -> 16.9.  They wait for all that
// was launched earlier in the threads that load.
// (The others do not let theirs start early: waiting beside them, the next prep kernel's blocks made a 2 x 128 x 128 x 3 heads
// call with k = 7 take 70 us instead of 59, others up to 6 % longer.)
template <typename... Params, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// The same for a prep kernel of few small blocks that may follow a kernel which lets it start early: with so much shared memory that an
// SM takes no more than its share of the blocks, or `Least` of them.  (They come while most SMs are still busy; without it they pile up, eight and more on
// the first few SMs that come free, and wait and work there: a forward of 8 x 56 x 56, 3 heads, bf16 and one with heads of 64 in turn 28.3 us
// spread, 34.3 piled up, 31.2 without early starts.  By themselves forwards with a prep launch take the same either way.)
template <auto Kernel, unsigned Least = 1, typename... Args>
inline cudaError_t launch_spread(dim3 grid, int threads, cudaStream_t stream, Args... args) {
    constexpr int kMost = 224 * 1024, kOwn = 2048;         // of 228 KB; a block's own and the system's beside it
    static int sms[64] = {};                               // of each device, once the kernel is set up there
    int dev = 0, n = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64) n = sms[dev];
    if (n == 0) {
        e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (dev < 64) sms[dev] = n;
    }
    const unsigned blocks = grid.x * grid.y;
    unsigned share = (blocks + (unsigned)n - 1) / (unsigned)n;
    if (share < Least) share = Least;
    return launch_chained(Kernel, grid, threads, share > 8 ? 0 : kMost / share - kOwn, stream, args...);
}

// Launchers.  Each returns cudaGetLastError() of its launch(es).
cudaError_t launch_direct(const Problem& p, cudaStream_t stream);
bool direct_supports(int head_dim, int ksize);

// STRIP variant: generic fp32 path with transposed weights (strip_workspace_bytes, written by the
// prep launch of every forward) and four pixels per warp.
bool strip_supports(int head_dim, int ksize);
size_t strip_workspace_bytes(int heads, int head_dim, int ksize);
cudaError_t launch_strip_prep(const Problem& p, void* workspace, cudaStream_t stream);
cudaError_t launch_strip_main(const Problem& p, const void* workspace, cudaStream_t stream);

// MMA variant.  `workspace` holds the re-laid-out weights (mma_workspace_bytes), written by the
// prep launch and read by the main launch on the same stream.  mma_setup must have succeeded once
// on the device before the first main launch.
bool mma_supports(slide_attn_dtype dtype, int head_dim, int ksize);
size_t mma_workspace_bytes(int heads);
cudaError_t mma_setup();
cudaError_t launch_mma_prep(const Problem& p, void* workspace, cudaStream_t stream);
cudaError_t launch_mma_main(const Problem& p, const void* workspace, int* d_status, cudaStream_t stream);


// UMMA_TS variant: both contractions on tcgen05 with their A operands in tensor memory.  The CTAs of the main launch lay out
// their head's weights themselves, or copy in what a prep launch left in `workspace` (umma_ts_workspace_bytes; null: none did).
bool umma_ts_supports(slide_attn_dtype dtype, int head_dim, int ksize);
cudaError_t umma_ts_setup();
size_t umma_ts_workspace_bytes(int heads);
cudaError_t launch_umma_ts_prep(const Problem& p, void* workspace, cudaStream_t stream);
cudaError_t launch_umma_ts(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream);

// UMMA_SPLIT variant: fp32 arithmetic on tcgen05 through exact splits (k = 3, head_dim 16, 32 or 64, both dtypes).  `workspace` as
// for UMMA_TS.
bool umma_split_supports(int head_dim, int ksize);
size_t umma_split_workspace_bytes(int heads, int head_dim);
bool umma_split_builds_images(int B, int H, int W, int heads, int num_sms);      // null is the better workspace
cudaError_t launch_umma_split_prep(const Problem& p, void* workspace, cudaStream_t stream);
cudaError_t launch_umma_split(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream);

// Fixed-shift fast path: plain k x k local attention for weights that are exactly the one-hot shift
// kernels (head_dim 32, k <= 9, fp32 or bf16).  launch_shift_check sets the status word to 2 when a
// weight differs from the one-hot kernel.
bool shift_supports(int head_dim, int ksize);
cudaError_t launch_shift_check(const Problem& p, int* d_status, cudaStream_t stream);
cudaError_t launch_shift(const Problem& p, int* d_status, cudaStream_t stream);
cudaError_t launch_shift_mma(const Problem& p, int* d_status, cudaStream_t stream);       // bf16, k = 5, 7, 9

// Backward pass (head_dim 32, k = 1 or 3, both dtypes): gradients of the forward's inputs.
struct BackwardArgs {
    const void* dout;    // [B][H][W][heads][head_dim], the problem's dtype
    void* dq;            // same shape and dtype
    void* dk;
    void* dv;
    float* dwk;          // [C][k*k][k*k]
    float* dwv;
    float* dbias;        // [heads][k*k] or nullptr
};
bool backward_supports(int head_dim, int ksize);
// Scratch: none for k = 1.  `compact` (k = 3): for half of the intermediate results only; the others lie in dv until it is written.
size_t backward_workspace_bytes(int B, int H, int W, int heads, int ksize, bool compact);
cudaError_t launch_backward(const Problem& p, const BackwardArgs& ga, void* ws, bool compact, int* d_status,
                            int num_sms, cudaStream_t stream);

// MMA_WIDE variant: general weights with large windows on tcgen05 (bf16, head_dim 32, k = 3, 5, 7, 9); a prep
// launch writes the weights as shared-memory images into `workspace`.
bool mma_wide_supports(slide_attn_dtype dtype, int head_dim, int ksize);
size_t mma_wide_workspace_bytes(int heads, int ksize);
cudaError_t launch_mma_wide_prep(const Problem& p, void* workspace, cudaStream_t stream);
cudaError_t launch_mma_wide(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream);

// TILE variant: generic weights, CUDA cores, TMA-staged halo tiles (head_dim 32, k <= 9, both dtypes).
// Reads the transposed weights that launch_strip_prep writes.
bool tile_supports(int head_dim, int ksize);
cudaError_t launch_tile(const Problem& p, const void* workspace, int* d_status, cudaStream_t stream);

// Projections of a block (Eq. 1 / Eq. 3) as a tcgen05 GEMM: y[i] = x w[i] for nmat row-major fp32 [c_in][c_out]
// matrices, x and y bf16 with channels contiguous.
bool proj_supports(int c_in, int c_out);
// `image`: w as launch_proj_prep laid it out (proj_image_bytes; two sets of matrices per launch), or null.
bool proj_wants_image(long long rows, int c_in, int c_out, int nmat, int num_sms);
size_t proj_image_bytes(int c_in, int c_out, int nmat);
cudaError_t launch_proj_prep(const float* wa, int nmat_a, void* image_a, const float* wb, int nmat_b, void* image_b, int c_in, int c_out, cudaStream_t stream);
// `early`: the kernel behind may start before this one is complete.
cudaError_t launch_proj(const void* x, long long rows, int c_in, const float* w, const void* image, int c_out, int nmat,
                        void* const* y, bool early, int* d_status, int num_sms, cudaStream_t stream);

}  // namespace slide_attn
