// Weight gradients of the backward pass for k = 3, bf16 storage (head_dim 32), on tcgen05:
//
//   dwk[c,s,t] = scale * sum over pixels of dl[s] (q[c] k_t[c])        dwv[c,s,t] = sum of a[s] (g[c] v_t[c])
//
// A matrix product over the pixels with the elementwise products as its left operand: rows (tap, channel), M = 128 = four taps
// x 32 channels, K = 16 pixels (2 rows x 8 columns), N = 32 columns of a split row (upper, middle and lower 8 bits of the fp32
// dl or a).  The products are exact as hi + lo, so nothing is rounded but the sums.  Five left operands cover both sides:
// taps 0 - 3 and 4 - 7 of the keys, the same of the values, and tap 8 of both (which meets dl and a).
//
//   left    products from registers to tensor memory: one transposing ldmatrix of a tile's channel planes (eight channels, 16
//           bytes a pixel) IS a 16-channel x 16-pixel fragment, at any tap's offset
//   right   the split rows as they lie in memory and as TMA brings them: 64 bytes a pixel, pieces swizzled by the column, which
//           is the 64-byte swizzle of an operand whose N index is contiguous
//   sums    the tensor core truncates when it accumulates, so after every chunk of 32 pixels the accumulators move to fp32
//           registers, and within one the lower parts come first: two truncations at full magnitude (after two chunks, in any
//           order: eight, error of dwk against 64 bits at 4 x 56 x 56 x 3 3.6e-7, so 2.3e-7, with fp32 FMAs 2.7e-7; 9 us less)
//
// Persistent, one CTA per SM and one head per CTA.  Sixteen compute warps = quadrant of tensor memory (tap mod 4) x side x
// 16-channel half, an MMA thread and a TMA thread.  Tiles of 4 rows x up to 56 columns + halo in two stages; a chunk = 4 rows x 8
// columns.  Bound by latency and instruction issue (50 M warp instructions at 64 x 56 x 56, 3 heads, in 46 % of the slots at 1.79 GHz:
// products, their splits and the reading of the accumulators): 410 us with fp32 FMAs on the CUDA cores, 134 on mma.sync, 106 here.
// Tensor-memory columns: six accumulators of 32, then two chunk buffers of [operand][16-pixel step][hi, lo: 8 each].
#include "bwd_common.cuh"
#include "split.cuh"

namespace slide_attn {

namespace {

constexpr int kHeadDim = 32, kK2 = 9, kTH = 4, kMaxW = 56;
constexpr int kComputeWarps = 16, kMmaWarp = kComputeWarps, kTmaWarp = kMmaWarp + 1;
constexpr int kThreads = (kTmaWarp + 1) * 32;
constexpr int kPlanes = 4;
constexpr float kTruncation = 7.3e-8f;                   // what two truncations take off on average (one: 4.3e-8, team.cuh)
constexpr uint32_t kColA = 192, kChunkCols = 160;
constexpr uint32_t kSumBytes = 6u * 128u * 32u * 4u;     // the CTA's sums at its end, [accumulator][row][32 columns]

struct Layout {
    uint32_t halo_plane, tile_plane, k_off, v_off, q_off, g_off, split_off, split_side, stage, tx_bytes;
};
__host__ __device__ inline Layout layout(int tw) {
    const uint32_t halo = (uint32_t)((kTH + 2) * (tw + 2)) * 16u, tile = (uint32_t)(kTH * tw) * 16u;
    auto up = [](uint32_t x, uint32_t to) { return (x + to - 1) / to * to; };
    Layout L;
    L.halo_plane = up(halo, 128); L.tile_plane = up(tile, 128);
    L.k_off = 0; L.v_off = kPlanes * L.halo_plane; L.q_off = 2 * kPlanes * L.halo_plane; L.g_off = L.q_off + kPlanes * L.tile_plane;
    L.split_off = up(L.g_off + kPlanes * L.tile_plane, 512);          // the swizzle's period
    L.split_side = (uint32_t)(kTH * tw) * 64u;
    L.stage = up(L.split_off + 2 * L.split_side, 512);
    L.tx_bytes = 2 * kPlanes * (halo + tile) + 2 * L.split_side;
    return L;
}
uint32_t smem_bytes(int tw) {
    const uint32_t stages = 2 * layout(tw).stage;
    return (stages > kSumBytes ? stages : kSumBytes) + 128 + 512;     // + barriers + alignment slack
}

struct WeightParams {
    float* dwk;
    float* dwv;
    int* status;
    int B, H, W, heads;
    int tw, tiles_x, tiles_y;
    float scale;
};

// Descriptor of 16 pixels x 32 columns: 64-byte rows, 64-byte swizzle, N contiguous; `next`: bytes to the second eight pixels.
__device__ __forceinline__ uint64_t rows_desc(uint32_t smem_addr, uint32_t next) {
    return (uint64_t)((smem_addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(next >> 4) << 32) | (1ull << 46) | (4ull << 61);
}
constexpr uint32_t kIdescNContiguous = 1u << 16;

__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}

// barriers: stage full / empty, chunk full / free, accumulators complete / read
enum : int { kFull = 0, kEmpty = 2, kAFull = 4, kAFree = 6, kDone = 8, kRead = 9, kBars = 10 };

__global__ void __launch_bounds__(kThreads, 1)
bwd_weight_umma_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                       const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_g,
                       const __grid_constant__ CUtensorMap map_dl, const __grid_constant__ CUtensorMap map_a, const WeightParams P)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((512u - (smem_u32(smem_raw) & 511u)) & 511u);
    const Layout L = layout(P.tw);
    const uint32_t stages = 2 * L.stage, bar0 = smem_u32(smem) + (stages > kSumBytes ? stages : kSumBytes);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    unsigned char* tmem_slot = smem + (bar0 - smem_u32(smem)) + 8 * kBars;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int h = blockIdx.x % P.heads, rank = blockIdx.x / P.heads, nrank = (int)gridDim.x / P.heads;
    const int tiles = P.B * P.tiles_y * P.tiles_x;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init_only(bar(kFull + i), 1); mbar_init_only(bar(kEmpty + i), kComputeWarps + 1);
            mbar_init_only(bar(kAFull + i), kComputeWarps); mbar_init_only(bar(kAFree + i), 1);
        }
        mbar_init_only(bar(kDone), 1);
        mbar_init_only(bar(kRead), kComputeWarps);
        mbar_init_fence();
    }
    if (warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *reinterpret_cast<const volatile uint32_t*>(tmem_slot);
    bool ok = true;
    auto columns = [&](int tile) { const int x0 = tile % P.tiles_x * P.tw; return min(P.tw, P.W - x0); };

    float sum[3][16];                                                 // of a compute warp: quarter warp / 4 of its quadrant's columns
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int c = 0; c < 16; ++c) sum[i][c] = 0.f;
    const int wq = warp & 3, part = (warp >> 2) & 3;

    if (warp == kTmaWarp) {
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
                if (!mbar_wait(bar(kEmpty + st), ((uint32_t)(it >> 1) & 1u) ^ 1u)) { ok = false; break; }
                mbar_expect_tx(bar(kFull + st), L.tx_bytes);
                tma_load_4d(stage + L.split_off, &map_dl, bar(kFull + st), h * 32, x0, y0, b);
                tma_load_4d(stage + L.split_off + L.split_side, &map_a, bar(kFull + st), h * 32, x0, y0, b);
#pragma unroll
                for (int pl = 0; pl < kPlanes; ++pl) {
                    const int c0 = h * kHeadDim + pl * 8;
                    tma_load_4d(stage + L.k_off + pl * L.halo_plane, &map_k, bar(kFull + st), c0, x0 - 1, y0 - 1, b);
                    tma_load_4d(stage + L.v_off + pl * L.halo_plane, &map_v, bar(kFull + st), c0, x0 - 1, y0 - 1, b);
                    tma_load_4d(stage + L.q_off + pl * L.tile_plane, &map_q, bar(kFull + st), c0, x0, y0, b);
                    tma_load_4d(stage + L.g_off + pl * L.tile_plane, &map_g, bar(kFull + st), c0, x0, y0, b);
                }
            }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        uint32_t leader;
        if (elect_one(leader)) {
            constexpr uint32_t id_hi = umma_idesc_bf16(128, 32) | kIdescNContiguous, id_lo = id_hi | kIdescNegateA;
            int it = 0, n = 0;                                       // tiles, chunks so far
            for (int tile = rank; ok && tile < tiles; tile += nrank, ++it) {
                const int st = it & 1, gx = columns(tile);
                if (!mbar_wait(bar(kFull + st), (uint32_t)(it >> 1) & 1u)) { ok = false; break; }
                const uint32_t rows = smem_u32(smem) + (uint32_t)st * L.stage + L.split_off;
                for (int c = 0; c < gx; c += 8, ++n) {
                    const int ab = n & 1;
                    if (n > 0 && !mbar_wait(bar(kRead), (uint32_t)(n - 1) & 1u)) { ok = false; break; }
                    if (!mbar_wait(bar(kAFull + ab), (uint32_t)(n >> 1) & 1u)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t a = tmem + kColA + (uint32_t)ab * kChunkCols;
                    for (int part = 1; part >= 0; --part)            // the lower parts of the products first
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks) {
                            const uint32_t at = rows + (uint32_t)(2 * ks * P.tw + c) * 64u;
                            const uint64_t dl = rows_desc(at, (uint32_t)P.tw * 64u), aw = rows_desc(at + L.split_side, (uint32_t)P.tw * 64u);
                            const uint32_t keep = part == 0 || ks != 0 ? 1u : 0u;
#pragma unroll
                            for (int i = 0; i < 6; ++i)              // accumulator i: operand i, or the fifth one for the last two
                                umma_bf16_ts(tmem + 32 * i, a + 32u * (uint32_t)(i < 5 ? i : 4) + 16u * ks + 8u * part, i < 2 || i == 4 ? dl : aw, part ? id_lo : id_hi, keep);
                        }
                    umma_commit(bar(kAFree + ab));
                    umma_commit(bar(kDone));
                }
                if (ok) umma_commit(bar(kEmpty + st));               // its rows have been read
            }
            // no commit on its way when the block leaves
            if (ok) { ok = wait_last_phases(bar(kAFree), 2, n); ok = wait_last_phases(bar(kEmpty), 2, it) && ok; }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else {
        const int side = part & 1, half = part >> 1;
        const uint32_t quad = tmem + ((uint32_t)(32 * wq) << 16), mine = quad + ((uint32_t)(16 * half) << 16);
        const bool ninth = wq == side;                               // tap 8: rows 0 - 31 the keys, 32 - 63 the values
        const int HW = P.tw + 2;
        // lane i of an ldmatrix: pixel i % 8 of row i / 16, channels 8 (i / 8 % 2) ..
        const uint32_t plane = (uint32_t)(2 * half + ((lane >> 3) & 1)), row = (uint32_t)(lane >> 4), col = (uint32_t)(lane & 7);
        const uint32_t x_off = (side ? L.g_off : L.q_off) + plane * L.tile_plane + (row * (uint32_t)P.tw + col) * 16u;
        const uint32_t y_off = (side ? L.v_off : L.k_off) + plane * L.halo_plane + (row * (uint32_t)HW + col) * 16u;
        const uint32_t t0 = (uint32_t)(wq / 3 * HW + wq % 3) * 16u, t1 = (uint32_t)((wq + 4) / 3 * HW + (wq + 4) % 3) * 16u,
                       t2 = (uint32_t)(2 * HW + 2) * 16u;
        int it = 0, n = 0;
        auto drain = [&](int chunk) -> bool {
            if (!warp_wait(bar(kDone), (uint32_t)chunk & 1u)) return false;
            tc_fence_after_sync();
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int idx = part + 4 * i;                        // 16 columns of accumulator idx / 2
                if (i == 2 && wq != (idx >= 10 ? 1 : 0)) continue;   // the last two hold tap 8 in one quadrant each
                float v[16];
                tmem_ld_32x32b_x16(quad + 16 * idx, v);
#pragma unroll
                for (int c = 0; c < 16; c += 2) fadd2(sum[i][c], sum[i][c + 1], v[c], v[c + 1]);
            }
            tc_fence_before_sync();
            __syncwarp();
            mbar_arrive_lane0(bar(kRead), lane);
            return true;
        };
        for (int tile = rank; ok && tile < tiles; tile += nrank, ++it) {
            const int st = it & 1, gx = columns(tile);
            if (!warp_wait(bar(kFull + st), (uint32_t)(it >> 1) & 1u)) { ok = false; break; }
            const uint32_t stage = smem_u32(smem) + (uint32_t)st * L.stage;
            uint32_t xa = stage + x_off, ya = stage + y_off;
            for (int c = 0; c < gx; c += 8, ++n, xa += 128, ya += 128) {
                const int ab = n & 1;
                if (!warp_wait(bar(kAFree + ab), ((uint32_t)(n >> 1) & 1u) ^ 1u)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t a = mine + kColA + (uint32_t)ab * kChunkCols;
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    uint32_t x[4], nx[4];
                    split::ldmatrix_x4_trans(xa + (uint32_t)(2 * ks * P.tw) * 16u, x[0], x[1], x[2], x[3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) nx[i] = x[i] ^ 0x80008000u;
                    auto tap = [&](uint32_t off, uint32_t op) {
                        uint32_t y[4], r[8];
                        split::ldmatrix_x4_trans(ya + off + (uint32_t)(2 * ks * HW) * 16u, y[0], y[1], y[2], y[3]);
#pragma unroll
                        for (int i = 0; i < 4; ++i) split::product2n(x[i], nx[i], y[i], r[i], r[4 + i]);
                        tmem_st_16x128b_x4(a + 32u * op + 16u * ks, r);
                    };
                    tap(t0, (uint32_t)(2 * side));
                    tap(t1, (uint32_t)(2 * side + 1));
                    if (ninth) tap(t2, 4u);
                }
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                mbar_arrive_lane0(bar(kAFull + ab), lane);
                // the sums of the chunk before: complete while this one was made
                if (n > 0 && !drain(n - 1)) { ok = false; break; }
            }
            __syncwarp();
            if (ok) mbar_arrive_lane0(bar(kEmpty + st), lane);
        }
        if (ok && n > 0) ok = drain(n - 1);
        if (!ok && lane == 0) atomicExch(P.status, 1);
    }
    tc_fence_before_sync();
    __syncthreads();                                                 // every load has been waited for: the stages are free
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
    float* s_sum = reinterpret_cast<float*>(smem);
    if (warp < kComputeWarps) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int idx = part + 4 * i;
            float* dst = s_sum + ((idx >> 1) * 128 + 32 * wq + lane) * 32 + (idx & 1) * 16;
#pragma unroll
            for (int c = 0; c < 16; c += 4) *reinterpret_cast<float4*>(dst + c) = make_float4(sum[i][c], sum[i][c + 1], sum[i][c + 2], sum[i][c + 3]);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kHeadDim * kK2 * kK2; i += kThreads) {
        const int sd = i >= kHeadDim * kK2 * kK2, rem = sd ? i - kHeadDim * kK2 * kK2 : i;
        const int ch = rem / (kK2 * kK2), st = rem - ch * kK2 * kK2;
        const int s = st / kK2, t = st - s * kK2;
        const float* p = s_sum + (t < 8 ? ((2 * sd + (t >> 2)) * 128 + 32 * (t & 3) + ch) : ((4 + sd) * 128 + 32 * sd + ch)) * 32 + s;
        const float v = fmaf(kTruncation, p[0], p[0] + (p[9] + p[18]));
        atomicAdd((sd ? P.dwv : P.dwk) + (size_t)(h * kHeadDim) * kK2 * kK2 + rem, sd ? v : v * P.scale);
    }
}

}  // namespace

cudaError_t launch_bwd_weight_umma(const Problem& p, const BackwardArgs& ga, const BwdScratch& ws, int* d_status, int num_sms, cudaStream_t stream) {
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !done[dev]) {
        e = cudaFuncSetAttribute(bwd_weight_umma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes(kMaxW));
        if (e != cudaSuccess) return e;
        if (dev < 64) done[dev] = true;
    }
    // the tile width (a multiple of 8) that covers the map with the fewest columns, the widest of those
    int tw = 8, cover = 1 << 30;
    for (int t = 8; t <= kMaxW; t += 8) {
        const int c = (p.W + t - 1) / t * t;
        if (c <= cover) { cover = c; tw = t; }
    }
    WeightParams P;
    P.dwk = ga.dwk; P.dwv = ga.dwv; P.status = d_status;
    P.B = p.B; P.H = p.H; P.W = p.W; P.heads = p.heads;
    P.tw = tw; P.tiles_x = (p.W + tw - 1) / tw; P.tiles_y = (p.H + kTH - 1) / kTH;
    P.scale = 1.f / sqrtf((float)kHeadDim);
    const int C = p.heads * kHeadDim;
    CUtensorMap mq, mk, mv, mg, mdl, ma;
    if (!make_tile_map(&mq, p.q, 2, p.B, p.H, p.W, C, 8, tw, kTH) || !make_tile_map(&mg, ga.dout, 2, p.B, p.H, p.W, C, 8, tw, kTH) ||
        !make_tile_map(&mk, p.k, 2, p.B, p.H, p.W, C, 8, tw + 2, kTH + 2) || !make_tile_map(&mv, p.v, 2, p.B, p.H, p.W, C, 8, tw + 2, kTH + 2) ||
        !make_tile_map(&mdl, ws.rows_dl, 2, p.B, p.H, p.W, C, 32, tw, kTH) || !make_tile_map(&ma, ws.rows_a, 2, p.B, p.H, p.W, C, 32, tw, kTH))
        return cudaErrorInvalidValue;
    const long long tiles = (long long)P.tiles_x * P.tiles_y * p.B;
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    long long per_head = num_sms / p.heads;                          // one CTA per SM, all heads alike
    if (per_head > tiles) per_head = tiles;
    if (per_head < 1) per_head = 1;
    return launch_chained(bwd_weight_umma_kernel, dim3((unsigned)(per_head * p.heads)), kThreads, smem_bytes(tw), stream, mq, mk, mv, mg, mdl, ma, P);
}

}  // namespace slide_attn
