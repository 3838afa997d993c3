// Shared by the backward kernels for k = 3: what they are launched with.
#pragma once
#include "common.cuh"

namespace slide_attn {

// Scratch of a backward pass with k = 3: the split rows (64 bytes, team.cuh) of the attention weights and of the logit gradients,
// [pixel][head], then the weight images of every head.  `compact`: the latter rows lie in dv's memory instead.
struct BwdScratch {
    unsigned char* rows_dl;
    unsigned char* rows_a;
    unsigned char* images;
};
size_t bwd_team_workspace_bytes(int B, int H, int W, int heads, bool compact);
BwdScratch bwd_scratch(void* ws, bool compact, void* dv, int B, int H, int W, int heads);

// point: clears the weight and bias gradients and builds the images, then dq, dbias and the split rows; gather: dk and dv from the split
// rows, behind everything else that reads them.
enum class BwdPass { point, gather };
cudaError_t launch_bwd_team(BwdPass what, const Problem& p, const BackwardArgs& ga, const BwdScratch& ws, int* d_status, int num_sms, cudaStream_t stream);
// dwk, dwv from the split rows: bf16 on tcgen05, fp32 on mma.sync.
cudaError_t launch_bwd_weight_umma(const Problem& p, const BackwardArgs& ga, const BwdScratch& ws, int* d_status, int num_sms, cudaStream_t stream);
cudaError_t launch_bwd_weight_mma(const Problem& p, const BackwardArgs& ga, const BwdScratch& ws, int* d_status, int num_sms, cudaStream_t stream);

}  // namespace slide_attn
