// Weight gradients of the backward pass for k = 3, fp32 storage (head_dim 32), on mma.sync (bf16: bwd_weight_umma_kernel):
//
//   dwk[c,s,t] = scale * sum over pixels of dl[s] (q[c] k_t[c])        dwv[c,s,t] = sum of a[s] (g[c] v_t[c])
//
// For one tap t and one side this is a matrix product over the pixels: [channels x pixels] . [pixels x slots],
// with the elementwise products as the left operand.  mma.sync.m16n8k16, M = 16 channels, K = 16 pixels (2 rows
// x 8 columns), N = 32 columns of a split row: the nine slots three times, the upper, middle and lower 8 bits of the
// fp32 dl (a).  The products are split into hi + mid + lo too; the pairs below 2^-24 are left out (hi meets all four
// 8-column tiles, mid the first three, lo the first two).
//
// Persistent, one CTA per SM and one head per CTA.  Twelve compute warps = side x 16-channel half x tap row,
// three per scheduler; a warp keeps the sums of its three taps in registers over all its tiles.  The tensor core
// truncates when it accumulates, so the columns that hold upper parts are added up in fp32 registers after every pixel group, and
// within one the smallest products come first: one truncation at full magnitude (after four groups, largest first: twelve, error of
// dwv against 64 bits 4.4e-7, so 1.8e-7, with fp32 FMAs 2.5e-7; the same time).  Tiles (4 rows x up to 32 columns + halo) come by TMA into
// two stages, in planes of 16 channels (four pixels x eight channel pairs = 256 contiguous bytes: no bank conflict).
//
// Bound by the mma.sync pipe and the CUDA-core work beside it, which hardly overlap (measured: 8 cycles per MMA and
// scheduler, and each packed bf16 multiply or fp32 add next to it adds 0.75 - 1.5): 324 MMAs per 16 pixels of a head.
// 2 x 128 x 128, 3 heads: 76 us with fp32 FMAs (lane = channel, 2 x 81 sums in registers), 45 us here.
#include "bwd_common.cuh"
#include "split.cuh"

namespace slide_attn {

namespace {

using namespace split;

constexpr int kHeadDim = 32;
constexpr int kK2 = 9;
constexpr int kTH = 4;                         // tile rows
constexpr int kComputeWarps = 12;
constexpr int kThreads = (kComputeWarps + 1) * 32;
constexpr float kTruncation = 4.3e-8f;         // what one truncation takes off on average (team.cuh): half of 2^-23 / (2 ln 2)
constexpr uint32_t kSumBytes = 2u * kK2 * kHeadDim * 32u * 4u;        // the CTA's sums at its end, [side][tap][channel][32 columns]

constexpr int kMaxW = 32;                      // tile columns
constexpr int kPlanes = 2;                     // planes of 16 channels
constexpr uint32_t kPixel = 64;                // bytes of a pixel in a plane

// Stage layout for tiles of tw columns (bytes); the channel planes of a tensor follow each other.
struct WLayout {
    uint32_t halo_plane, tile_plane;           // one plane with halo (k, v), without (q, g)
    uint32_t k_off, v_off, q_off, g_off;
    uint32_t split_off, split_side;            // dl columns, then a columns: [pixel][32] bf16
    uint32_t stage;                            // bytes of a stage
    uint32_t tx_bytes;
};
__host__ __device__ inline WLayout w_layout(int tw) {
    constexpr uint32_t np = kPlanes, pb = kPixel;
    auto up = [](uint32_t x) { return (x + 127u) & ~127u; };
    WLayout L;
    const uint32_t halo = (uint32_t)((kTH + 2) * (tw + 2)) * pb, tile = (uint32_t)(kTH * tw) * pb;
    L.halo_plane = up(halo); L.tile_plane = up(tile);
    L.k_off = 0; L.v_off = np * L.halo_plane; L.q_off = 2 * np * L.halo_plane; L.g_off = L.q_off + np * L.tile_plane;
    L.split_off = L.g_off + np * L.tile_plane;
    L.split_side = (uint32_t)(kTH * tw) * 64u;
    L.stage = L.split_off + 2 * L.split_side;
    L.tx_bytes = 2 * np * (halo + tile) + 2 * L.split_side;
    return L;
}

uint32_t w_smem_bytes(int tw) {
    const uint32_t stages = 2 * w_layout(tw).stage;
    return (stages > kSumBytes ? stages : kSumBytes) + 64 + 128;      // + barriers + alignment slack
}

struct WParams {
    float* dwk;
    float* dwv;
    int* status;
    int B, H, W, heads;
    int tw, tiles_x, tiles_y;
    float scale;
};

// One 16-pixel (2 rows x 8 columns), 16-channel operand tile in registers: the values of channels 2g, 2g + 1 of the lane's
// four pixels.  `offset`: where a lane reads in a tile whose planes are `plane` bytes apart; `col`: which column of the group the K index
// k (of its row's eight) is; `channel`: which of the 16 channels the row is.
struct Frag {
    float2 a[4];
    static __device__ __forceinline__ uint32_t offset(int lane, int half, uint32_t plane) {
        return (uint32_t)half * plane + (uint32_t)(lane & 3) * kPixel + (uint32_t)(lane >> 2) * 8u;
    }
    static __device__ __forceinline__ int col(int k) { return (k & 1) * 4 + (k >> 1); }
    static __device__ __forceinline__ int channel(int row) { return 2 * (row & 7) + (row >> 3); }
    __device__ __forceinline__ void load(uint32_t p, uint32_t pitch) {
        a[0] = lds_f2(p); a[1] = lds_f2(p + 4 * kPixel);
        a[2] = lds_f2(p + pitch); a[3] = lds_f2(p + pitch + 4 * kPixel);
    }
};

// sum += (x . y) times the split columns b[tile][2]
__device__ __forceinline__ void accumulate(float (&sum)[4][4], const Frag& x, const Frag& y, const uint32_t (&b)[4][2]) {
    float2 p[4];
    uint32_t a[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = mul2(x.a[i], y.a[i]);
#pragma unroll
    for (int part = 0; part < 3; ++part) {
        a[part][0] = pack_upper(p[0].x, p[1].x); a[part][1] = pack_upper(p[0].y, p[1].y);
        a[part][2] = pack_upper(p[2].x, p[3].x); a[part][3] = pack_upper(p[2].y, p[3].y);
        if (part < 2)
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = rest2(p[i]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {                                    // columns of upper (and some middle) parts
        float c[4];
        mma_bf16_c(c, a[2], b[j][0], b[j][1], 0.f, 0.f, 0.f, 0.f);
        mma_bf16(c, a[1], b[j][0], b[j][1]);
        mma_bf16(c, a[0], b[j][0], b[j][1]);
        fadd2(sum[j][0], sum[j][1], c[0], c[1]);
        fadd2(sum[j][2], sum[j][3], c[2], c[3]);
    }
    mma_bf16(sum[2], a[1], b[2][0], b[2][1]);
    mma_bf16(sum[2], a[0], b[2][0], b[2][1]);
    mma_bf16(sum[3], a[0], b[3][0], b[3][1]);
}

__global__ void __launch_bounds__(kThreads, 1)
bwd_weight_mma_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                      const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_g,
                      const __grid_constant__ CUtensorMap map_dl, const __grid_constant__ CUtensorMap map_a, const WParams P)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const WLayout L = w_layout(P.tw);
    const uint32_t stages = 2 * L.stage;
    const uint32_t bar0 = smem_u32(smem) + (stages > kSumBytes ? stages : kSumBytes);
    auto bar_full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
    auto bar_empty = [&](int s) { return bar0 + 16u + 8u * (uint32_t)s; };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;
    const int h = blockIdx.x % P.heads, rank = blockIdx.x / P.heads;
    const int nrank = (int)gridDim.x / P.heads;                      // the grid is a multiple of the heads
    const int tiles = P.B * P.tiles_y * P.tiles_x;
    const int HW = P.tw + 2;

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) { mbar_init_only(bar_full(s), 1); mbar_init_only(bar_empty(s), kComputeWarps); }
        mbar_init_fence();
    }
    __syncthreads();

    float sum[3][4][4];
    bool ok = true;
    const int side = warp / 6, half = (warp / 3) & 1, ty = warp % 3;  // of a compute warp

    if (warp >= kComputeWarps) {
        // ---- TMA thread --------------------------------------------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            grid_dependency_wait();                                  // the split rows come from an earlier kernel
            int it = 0;
            for (int tile = rank; tile < tiles; tile += nrank, ++it) {
                const int st = it & 1;
                int rest_ = tile;
                const int tx = rest_ % P.tiles_x; rest_ /= P.tiles_x;
                const int tyy = rest_ % P.tiles_y;
                const int b = rest_ / P.tiles_y;
                const int x0 = tx * P.tw, y0 = tyy * kTH;
                const uint32_t stage = smem_u32(smem) + (uint32_t)st * L.stage;
                if (it >= 2 && !mbar_wait(bar_empty(st), (uint32_t)(it / 2 - 1) & 1u)) { ok = false; break; }
                mbar_expect_tx(bar_full(st), L.tx_bytes);
                tma_load_4d(stage + L.split_off, &map_dl, bar_full(st), h * 32, x0, y0, b);
                tma_load_4d(stage + L.split_off + L.split_side, &map_a, bar_full(st), h * 32, x0, y0, b);
#pragma unroll
                for (int pl = 0; pl < kPlanes; ++pl) {
                    const int c0 = h * kHeadDim + pl * (32 / kPlanes);
                    tma_load_4d(stage + L.k_off + pl * L.halo_plane, &map_k, bar_full(st), c0, x0 - 1, y0 - 1, b);
                    tma_load_4d(stage + L.v_off + pl * L.halo_plane, &map_v, bar_full(st), c0, x0 - 1, y0 - 1, b);
                    tma_load_4d(stage + L.q_off + pl * L.tile_plane, &map_q, bar_full(st), c0, x0, y0, b);
                    tma_load_4d(stage + L.g_off + pl * L.tile_plane, &map_g, bar_full(st), c0, x0, y0, b);
                }
            }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else {
        // ---- products and sums ----------------------------------------------------------------------
#pragma unroll
        for (int t = 0; t < 3; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int x = 0; x < 4; ++x) sum[t][j][x] = 0.f;
        // lane i of the ldmatrix of the split columns: K index i % 8 of row (i / 8) % 2, 16-byte chunk i / 16 (+ 2)
        const int kcol = Frag::col(lane & 7);
        const uint32_t b_off = L.split_off + (uint32_t)side * L.split_side + (uint32_t)(((lane >> 3) & 1) * P.tw + kcol) * 64u;
        const uint32_t b_chunk0 = (((uint32_t)lane >> 4) ^ ((uint32_t)kcol >> 1)) << 4;
        const uint32_t b_chunk1 = ((2u + ((uint32_t)lane >> 4)) ^ ((uint32_t)kcol >> 1)) << 4;
        const uint32_t x_pitch = (uint32_t)P.tw * kPixel, y_pitch = (uint32_t)HW * kPixel;
        const uint32_t x_off = (side ? L.g_off : L.q_off) + Frag::offset(lane, half, L.tile_plane);
        const uint32_t y_off = (side ? L.v_off : L.k_off) + (uint32_t)ty * y_pitch + Frag::offset(lane, half, L.halo_plane);
        int it = 0;
        for (int tile = rank; tile < tiles; tile += nrank, ++it) {
            const int st = it & 1;
            int rest_ = tile;
            const int tx = rest_ % P.tiles_x; rest_ /= P.tiles_x;
            const int tyy = rest_ % P.tiles_y;
            const int gx = min(P.tw, P.W - tx * P.tw), gy = min(kTH, P.H - tyy * kTH);   // part of the tile inside the map
            const uint32_t stage = smem_u32(smem) + (uint32_t)st * L.stage;
            if (!__all_sync(0xffffffffu, mbar_wait(bar_full(st), (uint32_t)(it / 2) & 1u) ? 1 : 0)) { ok = false; break; }
            for (int r = 0; r < gy; r += 2) {
                uint32_t ba = stage + b_off + (uint32_t)(r * P.tw) * 64u;
                uint32_t xa = stage + x_off + (uint32_t)r * x_pitch, ya = stage + y_off + (uint32_t)r * y_pitch;
                for (int c = 0; c < gx; c += 8, ba += 8 * 64, xa += 8 * kPixel, ya += 8 * kPixel) {
                    uint32_t b[4][2];
                    ldmatrix_x4_trans(ba + b_chunk0, b[0][0], b[0][1], b[1][0], b[1][1]);
                    ldmatrix_x4_trans(ba + b_chunk1, b[2][0], b[2][1], b[3][0], b[3][1]);
                    Frag x, y[3];
                    x.load(xa, x_pitch);
#pragma unroll
                    for (int t = 0; t < 3; ++t) y[t].load(ya + t * kPixel, y_pitch);
#pragma unroll
                    for (int t = 0; t < 3; ++t) accumulate(sum[t], x, y[t], b);
                }
            }
            // the sums have taken in everything that was loaded: tile 0 of a tap its products and the first split columns, tile 2 the others
            uint32_t read = 0;
#pragma unroll
            for (int t = 0; t < 3; ++t) read |= __float_as_uint(sum[t][0][0]) | __float_as_uint(sum[t][2][0]);
            __syncwarp();
            mbar_arrive_lane0_after(bar_empty(st), lane, __uint_as_float(read), 0.f, (uint32_t)(P.H >> 31));
        }
    }
    if (!ok && lane == 0) atomicExch(P.status, 1);
    __syncthreads();                                                 // every load has been waited for: the stages are free
    float* s_sum = reinterpret_cast<float*>(smem);
    if (warp < kComputeWarps) {
#pragma unroll
        for (int t = 0; t < 3; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int ch = half * 16 + Frag::channel(g + 8 * (x >> 1));
                    s_sum[((side * kK2 + ty * 3 + t) * kHeadDim + ch) * 32 + 8 * j + 2 * tig + (x & 1)] = sum[t][j][x];
                }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kHeadDim * kK2 * kK2; i += kThreads) {
        const int sd = i >= kHeadDim * kK2 * kK2, rem = sd ? i - kHeadDim * kK2 * kK2 : i;
        const int ch = rem / (kK2 * kK2), st = rem - ch * kK2 * kK2;
        const int s = st / kK2, t = st - s * kK2;
        const float* p = s_sum + ((sd * kK2 + t) * kHeadDim + ch) * 32 + s;
        const float v = fmaf(kTruncation, p[0], p[0] + (p[9] + p[18]));
        atomicAdd((sd ? P.dwv : P.dwk) + (size_t)(h * kHeadDim) * kK2 * kK2 + rem, sd ? v : v * P.scale);
    }
}

}  // namespace

cudaError_t launch_bwd_weight_mma(const Problem& p, const BackwardArgs& ga, const BwdScratch& ws, int* d_status, int num_sms, cudaStream_t stream) {
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !done[dev]) {
        e = cudaFuncSetAttribute(bwd_weight_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)w_smem_bytes(kMaxW));
        if (e != cudaSuccess) return e;
        if (dev < 64) done[dev] = true;
    }
    // the tile width (a multiple of 8) that covers the map with the fewest columns, the widest of those
    int tw = 8, cover = 1 << 30;
    for (int t = 8; t <= kMaxW; t += 8) {
        const int c = (p.W + t - 1) / t * t;
        if (c <= cover) { cover = c; tw = t; }
    }
    WParams P;
    P.dwk = ga.dwk; P.dwv = ga.dwv; P.status = d_status;
    P.B = p.B; P.H = p.H; P.W = p.W; P.heads = p.heads;
    P.tw = tw; P.tiles_x = (p.W + tw - 1) / tw; P.tiles_y = (p.H + kTH - 1) / kTH;
    P.scale = 1.f / sqrtf((float)kHeadDim);
    const int Ctot = p.heads * kHeadDim, es = (int)sizeof(float), bc = kHeadDim / kPlanes;
    CUtensorMap mq, mk, mv, mg, mdl, ma;
    if (!make_tile_map(&mq, p.q, es, p.B, p.H, p.W, Ctot, bc, tw, kTH) ||
        !make_tile_map(&mg, ga.dout, es, p.B, p.H, p.W, Ctot, bc, tw, kTH) ||
        !make_tile_map(&mk, p.k, es, p.B, p.H, p.W, Ctot, bc, tw + 2, kTH + 2) ||
        !make_tile_map(&mv, p.v, es, p.B, p.H, p.W, Ctot, bc, tw + 2, kTH + 2) ||
        !make_tile_map(&mdl, ws.rows_dl, 2, p.B, p.H, p.W, Ctot, 32, tw, kTH) || !make_tile_map(&ma, ws.rows_a, 2, p.B, p.H, p.W, Ctot, 32, tw, kTH))
        return cudaErrorInvalidValue;
    const long long tiles = (long long)P.tiles_x * P.tiles_y * p.B;
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    long long per_head = num_sms / p.heads;                          // one CTA per SM, all heads alike
    if (per_head > tiles) per_head = tiles;
    if (per_head < 1) per_head = 1;
    return launch_chained(bwd_weight_mma_kernel, dim3((unsigned)(per_head * p.heads)), kThreads, w_smem_bytes(tw), stream, mq, mk, mv, mg, mdl, ma, P);
}

}  // namespace slide_attn
