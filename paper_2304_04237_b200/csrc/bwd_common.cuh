// Shared by the backward kernels: what they are launched with.
#pragma once
#include "common.cuh"

namespace slide_attn {

struct BwdParams {
    const float* wt;                 // transposed weights wk^T then wv^T, [slot][tap][C]
    const float* bias;
    void* dq;
    void* dk;
    void* dv;
    float* dwk;
    float* dwv;
    float* dbias;
    float* ws_a;                     // [pixel][head][k*k]
    float* ws_dl;
    int* status;
    int B, H, W, heads;
    int tiles_x, tiles_y;
    float scale;                     // 1 / sqrt(head_dim)
};

// dwk, dwv for k = 3 on the tensor cores; P as the point kernel was given it, a and dl already in its workspace.
cudaError_t launch_bwd_weight_mma(const Problem& p, const BackwardArgs& ga, const BwdParams& P, int num_sms, cudaStream_t stream);

}  // namespace slide_attn
