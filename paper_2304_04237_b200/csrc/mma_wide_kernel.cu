// MMA_WIDE variant: deformed (general) depthwise weights with LARGE windows on tensor cores (the
// paper's stated limitation, App. E-F: k > 3 costs "a huge increase on the inference time"): bf16,
// head_dim 32, k = 5, 7, 9 (k = 3 compiles too and serves as a cross-check).
//
// Arithmetic (Eq. 2 with Eq. 12 inside; w = E + D, E the one-hot shift of Eq. 11, D the remainder), both contractions on
// tcgen05 with their left operands in tensor memory:
//   P[p,(t,c)]  = q[p,c] k[p+off(t),c]                    packed bf16 multiplies -> tensor memory
//   L[p,s]     += sum_c P[p,(t,c)] D_k[c,s,t]             per tap M = 128, N = slots (rounded up to 16), K = 32
//   L[p,t]     += sum_c P[p,(t,c)]                        one-hot part: N = 16 columns around t against a column of ones, which
//                                                         a window sliding over [0 .. 0 1 0 .. 0] puts at any column
//   e[s]        = exp(L scale + bias - the largest of them), kept as e_hi + e_lo (two bf16)
//   A'[p,(t,c)] = sum_s e_hi[p,s] D_v[c,s,t] + (e_hi + e_lo)[p,t]          N = 32 per tap, K = slots; then K = 16 around t, twice
//   out[p,c]    = (sum_t A'[p,t,c] v[p+off(t),c]) / sum_s e[s]              packed fp32 FMAs
// The weights are divided by their sum at the end only: the largest e is 1, which bf16 holds exactly, whereas a normalised
// weight is rounded like any other (error of the result against 64 bits, 2 x 56 x 56 x 2, k = 7, one-hot weights + N(0, 0.21): 3.61e-3,
// with normalised weights 3.78e-3).
// 2 k^4 multiply-adds per pixel-channel go to the tensor cores; the CUDA cores keep 2 k^2.
//
// Persistent, one CTA per SM, one head per CTA; two teams of eight warps, each with its own block of 128 pixels = two TILES of
// 8 x 8 pixels.  Warps q and q + 4 of a team have quadrant q of tensor memory: rows 4 (q % 2) .. + 3 of tile q / 2, the first
// their upper two, the second their lower two; lane (g, tig) works on column g and channels 8 tig .. 8 tig + 7.  Tiles come by
// TMA with their halo (zero fill = the padding), K then V.  Five more warps: an MMA and a TMA thread per team; one for weights.
// The weights (2 x 32 k^4 bf16 per head, laid out by a prep kernel in the order they are used) stay in shared memory for
// k <= 5 (102 KB at k = 5), so the teams run independently and cover each other's hand-offs; for k >= 7 (400 KB, 1 MB) they are
// streamed from L2 through a ring that both teams read, 256 pixels per pass over them.
//
// Tensor-memory columns of a team (256): logits, later e (chunk of 16 slots: 8 columns e_hi, 8 e_lo, where its logits were), in
// the last N; below them the product groups, later the A' groups.  A group = up to GK (GV) taps of one tap column.
//
// A call: 64 x 56 x 56, 3 heads, k = 5: 273 us with mma.sync (every CUDA-core multiply beside it cost it pipe time, and every
// fragment was read from shared memory by every warp), 133 here (71 M warp instructions in 52 % of the issue slots at 1.70 GHz, tensor pipe
// 38 %); 2 x 128 x 128, 3 heads, k = 7: 137 and 60 us (39 and 40 %: three rounds for 2.6 blocks per team).
#include "common.cuh"
#include "ptx.cuh"

namespace slide_attn {

namespace {

constexpr int kHeadDim = 32;
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kTeams = 2, kTeamWarps = 8, kComputeWarps = kTeams * kTeamWarps;
constexpr int kMmaWarp = kComputeWarps, kTmaWarp = kMmaWarp + kTeams, kWeightWarp = kTmaWarp + kTeams;
constexpr int kThreads = (kWeightWarp + 1) * 32;
constexpr uint32_t kOnesBytes = 2 * 512;                 // [two 8-channel chunks][31 rows of 16 bytes], row 15 ones
constexpr uint32_t kUnitBytes = 4 * 10 * 128;            // [four groups of 8 columns][zeros, ones in k = 0 .. 7, zeros]
constexpr uint32_t kInvBytes = kTeams * 128 * 4;         // 1 / sum of the weights of each pixel
constexpr uint32_t kMaxSmem = 227 * 1024;

// barriers of a team, then those of the weights
enum : int { kPFull = 0, kPFree = 3, kLFull = 6, kAFull = 7, kDFull = 8, kDFree = 10, kFull = 12, kEmpty = 15, kTeamBars = 18 };
enum : int { kWFull = kTeams * kTeamBars, kWEmpty = kWFull + 3, kBars = kWEmpty + 3 };

constexpr int least(int a, int b) { return a < b ? a : b; }

template <int K>
struct Wide {
    static constexpr int K2 = K * K, R = K / 2;
    static constexpr int KS = (K2 + 15) / 16;            // K steps of the value side
    static constexpr int N = 16 * KS;                    // columns of the logits
    static constexpr bool resident = K <= 5;
    static constexpr int GK = K == 5 ? 5 : K == 7 ? 4 : 3, GV = K == 9 ? 2 : 3;
    static constexpr int NGK = (K + GK - 1) / GK, NGV = (K + GV - 1) / GV;
    static constexpr int PB = least(3, (256 - N) / (16 * GK)), DB = 2;
    static_assert(DB * 32 * GV <= 256 - N && PB >= 2, "tensor memory");
    static constexpr int HP = 8 + 2 * R;                 // edge of a tile with its halo
    static constexpr uint32_t plane = (uint32_t)(HP * HP * 64), slot = 2 * plane;
    static constexpr uint32_t tap = (uint32_t)(N * 64);  // weights of a tap, either side
    static constexpr uint32_t weights = 2u * K2 * tap;   // of a head
    static constexpr uint32_t chunk = (uint32_t)(GK > GV ? GK : GV) * tap;
    static constexpr uint32_t w_bytes = resident ? weights : 3 * chunk;
    static constexpr uint32_t misc = kOnesBytes + kUnitBytes + 336 + kInvBytes + 8u * kBars + 16;
    static constexpr int ring = least(3, (int)((kMaxSmem - w_bytes - misc - 128) / (kTeams * slot)));
    static_assert(ring >= 2, "the ring does not fit");
    static constexpr uint32_t w_off = (uint32_t)(kTeams * ring) * slot, ones_off = w_off + w_bytes, unit_off = ones_off + kOnesBytes,
                              bias_off = unit_off + kUnitBytes, inv_off = bias_off + 336, bar_off = inv_off + kInvBytes, tmem_off = bar_off + 8u * kBars,
                              total = tmem_off + 16 + 128;
};

// A walk over the 8 x 8 tiles of the maps from a given one in equal steps, by carries.
struct TileWalk {
    int b, y, x, db, dy, dx, tx, ty;
    __device__ __forceinline__ TileWalk(int tiles_x, int tiles_y, int first, int step) : tx(tiles_x), ty(tiles_y) {
        x = first % tx; y = first / tx % ty; b = first / tx / ty;
        dx = step % tx; dy = step / tx % ty; db = step / tx / ty;
    }
    __device__ __forceinline__ void next() {
        x += dx; y += dy; b += db;
        if (x >= tx) { x -= tx; ++y; }
        if (y >= ty) { y -= ty; ++b; }
    }
};

struct WideParams {
    const unsigned char* weights;    // [head][Wide::weights]
    const __nv_bfloat16* q;
    const float* bias;
    __nv_bfloat16* out;
    int* status;
    int H, W, heads;
    int tiles_x, tiles_y, tiles;
    float scale_log2e;
};

// Prep: fp32 [C][slot][tap] -> bf16, taps in the order o = dx K + dy (tap t = dy K + dx), first the key side, then the value side,
// one 16-byte item per thread.
//   key tap, item (j, n): k 8j .. 8j + 7 (channels in the order tcgen05.st lays the products out), column n = slot
//   value tap, item (n, j): column n (channel in the order tcgen05.ld hands them out), k 8j .. 8j + 7 = slots
template <int K>
__global__ void __launch_bounds__(256)
mma_wide_prep_kernel(const float* __restrict__ wk, const float* __restrict__ wv, unsigned char* __restrict__ img)
{
    using Wd = Wide<K>;
    constexpr int K2 = Wd::K2, N = Wd::N, per_tap = 4 * N;
    grid_dependency_wait();
    grid_launch_dependents();
    const int h = blockIdx.y;
    const float* wkh = wk + (size_t)h * kHeadDim * K2 * K2;
    const float* wvh = wv + (size_t)h * kHeadDim * K2 * K2;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < 2 * K2 * per_tap; i += gridDim.x * 256) {
        const int side = i >= K2 * per_tap, r = side ? i - K2 * per_tap : i;
        const int o = r / per_tap, item = r % per_tap, t = (o % K) * K + o / K;
        unsigned char* tap = img + (size_t)h * Wd::weights + (size_t)(side * K2 + o) * Wd::tap;
        float v[8];
        uint32_t at;
        if (side == 0) {
            const int n = item % N, j = item / N;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int kap = 8 * j + e, c = 8 * ((kap & 15) >> 2) + (kap & 3) + (kap >= 16 ? 4 : 0);
                v[e] = n < K2 ? wkh[((size_t)c * K2 + n) * K2 + t] - (n == t ? 1.f : 0.f) : 0.f;
            }
            at = (uint32_t)(j * N * 16 + n * 16);
        } else {
            const int n = item & 31, j = item >> 5, c = 8 * ((n & 7) >> 1) + 2 * (n >> 3) + (n & 1);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int s = 8 * j + e;
                v[e] = s < K2 ? wvh[((size_t)c * K2 + s) * K2 + t] - (s == t ? 1.f : 0.f) : 0.f;
            }
            at = (uint32_t)((n >> 3) * (2 * Wd::KS * 128) + j * 128 + (n & 7) * 16);
        }
        *reinterpret_cast<uint4*>(tap + at) = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    }
}

__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}

// Products of G taps (halo rows dy0 .. of column dx) for the lane's two pixels into tensor memory at `t`, 16 columns a tap.
template <int G, int HP>
__device__ __forceinline__ void store_products(uint32_t t, const unsigned char* src, const uint4 (&x)[2]) {
    uint4 y[G + 1];
#pragma unroll
    for (int r = 0; r <= G; ++r) y[r] = *reinterpret_cast<const uint4*>(src + r * HP * 64);
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const uint32_t r[8] = {hmul2_bf16(x[0].x, y[i].x), hmul2_bf16(x[0].y, y[i].y), hmul2_bf16(x[1].x, y[i + 1].x), hmul2_bf16(x[1].y, y[i + 1].y),
                               hmul2_bf16(x[0].z, y[i].z), hmul2_bf16(x[0].w, y[i].w), hmul2_bf16(x[1].z, y[i + 1].z), hmul2_bf16(x[1].w, y[i + 1].w)};
        tmem_st_16x256b_x2(t + 16 * i, r);
    }
}
// acc += the A' of G taps at `t` times their halo pixels.
template <int G, int HP>
__device__ __forceinline__ void sum_group(uint32_t t, const unsigned char* src, float (&acc)[2][8]) {
    uint32_t d[G][16];
#pragma unroll
    for (int i = 0; i < G; ++i) tmem_ld_16x256b_x4_nowait(t + 32 * i, d[i]);
    uint4 y[G + 1];
#pragma unroll
    for (int r = 0; r <= G; ++r) y[r] = *reinterpret_cast<const uint4*>(src + r * HP * 64);
    float f[G + 1][8];
#pragma unroll
    for (int r = 0; r <= G; ++r) {
        f[r][0] = bf16_lo(y[r].x); f[r][1] = bf16_hi(y[r].x); f[r][2] = bf16_lo(y[r].y); f[r][3] = bf16_hi(y[r].y);
        f[r][4] = bf16_lo(y[r].z); f[r][5] = bf16_hi(y[r].z); f[r][6] = bf16_lo(y[r].w); f[r][7] = bf16_hi(y[r].w);
    }
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < G; ++i) {
        tmem_pass(d[i]);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                ffma2(acc[r][2 * j], acc[r][2 * j + 1], __uint_as_float(d[i][4 * j + 2 * r]), __uint_as_float(d[i][4 * j + 2 * r + 1]),
                      f[r + i][2 * j], f[r + i][2 * j + 1]);
    }
}

// Softmax of the lane's pixel, whose N logits start at tensor-memory column `col`; leaves e_hi, e_lo in their place, returns 1 / sum.
template <int K>
__device__ __forceinline__ float softmax_in_place(uint32_t col, const float* s_bias, float scale_log2e) {
    using Wd = Wide<K>;
    constexpr int K2 = Wd::K2, KS = Wd::KS;
    constexpr bool keep = KS <= 2;                       // the logits stay in registers between the passes
    float l[keep ? KS : 1][16];
    auto load = [&](int j, float (&v)[16]) {
        tmem_ld_32x32b_x16(col + 16 * j, v);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (16 * j + i < K2) v[i] = fmaf(v[i], scale_log2e, s_bias[16 * j + i]);
    };
    // the largest of all slots first: a running one is -inf while all slots so far are masked by a bias of -inf, and exp2(-inf + inf)
    // is not a number
    // (k >= 7, unrolled: registers spill, 61.6 us instead of 60.0 at 2 x 128 x 128, 3 heads, k = 7)
    float m = -INFINITY, z = 0.f;
#pragma unroll (keep ? KS : 1)
    for (int j = 0; j < KS; ++j) {
        float (&v)[16] = l[keep ? j : 0];
        load(j, v);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (16 * j + i < K2) m = fmaxf(m, v[i]);
    }
#pragma unroll (keep ? KS : 1)
    for (int j = 0; j < KS; ++j) {
        float (&v)[16] = l[keep ? j : 0];
        if (!keep) load(j, v);
        uint32_t row[16];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float e0 = 16 * j + 2 * i < K2 ? fast_exp2(v[2 * i] - m) : 0.f, e1 = 16 * j + 2 * i + 1 < K2 ? fast_exp2(v[2 * i + 1] - m) : 0.f;
            z += e0; z += e1;
            row[i] = pack_bf16(e0, e1);
            row[8 + i] = pack_bf16(e0 - bf16_lo(row[i]), e1 - bf16_hi(row[i]));
        }
        tmem_st_32x32b_x16(col + 16 * j, row);
    }
    tmem_wait_st();
    return 1.f / z;
}

template <int K>
__global__ void __launch_bounds__(kThreads, 1)
mma_wide_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const WideParams P)
{
    using Wd = Wide<K>;
    constexpr int N = Wd::N, KS = Wd::KS, GK = Wd::GK, GV = Wd::GV, NGK = Wd::NGK, NGV = Wd::NGV, PB = Wd::PB, DB = Wd::DB, HP = Wd::HP, R = Wd::ring;
    constexpr uint32_t kColL = 256 - N;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const uint32_t bars = smem_u32(smem + Wd::bar_off);
    float* s_bias = reinterpret_cast<float*>(smem + Wd::bias_off);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int h = blockIdx.x % P.heads, rank = blockIdx.x / P.heads, nrank = (int)gridDim.x / P.heads;
    const int team_id = warp < kComputeWarps ? warp / kTeamWarps : (warp - kComputeWarps) % kTeams;
    const int blocks = (P.tiles + 1) >> 1, step = kTeams * nrank, first = team_id * nrank + rank;
    auto blocks_from = [&](int at) { return at < blocks ? (blocks - at + step - 1) / step : 0; };
    const int my_blocks = blocks_from(first), rounds = blocks_from(rank);            // rounds: of team 0, which has the most
    auto bar = [&](int i) { return bars + 8u * (uint32_t)(team_id * kTeamBars + i); };
    auto wbar = [&](int i) { return bars + 8u * (uint32_t)i; };

    if (threadIdx.x == 0) {
        for (int t = 0; t < kTeams; ++t) {
            auto init = [&](int i, uint32_t count) { mbar_init_only(bars + 8u * (uint32_t)(t * kTeamBars + i), count); };
            for (int i = 0; i < 3; ++i) { init(kPFull + i, kTeamWarps); init(kPFree + i, 1); init(kFull + i, 1); init(kEmpty + i, kTeamWarps); }
            init(kLFull, 1);
            init(kAFull, 4);
            for (int i = 0; i < 2; ++i) { init(kDFull + i, 1); init(kDFree + i, kTeamWarps); }
        }
        for (int i = 0; i < 3; ++i) { mbar_init_only(wbar(kWFull + i), 1); mbar_init_only(wbar(kWEmpty + i), kTeams); }
        mbar_init_fence();
    }
    for (int i = threadIdx.x; i < Wd::K2; i += kThreads) s_bias[i] = P.bias ? P.bias[h * Wd::K2 + i] * kLog2e : 0.f;
    for (uint32_t i = threadIdx.x; i < (kOnesBytes + kUnitBytes) / 4; i += kThreads) {
        uint32_t v = 0;
        if (i < kOnesBytes / 4) {
            if (((i * 4) & 511u) >> 4 == 15) v = kOnesBf16x2;
        } else {
            const uint32_t b = (i * 4 - kOnesBytes) % 1280u, core = b >> 7, k = (b & 15u) >> 1;      // k, k + 1 of a row
            if (core >= 1 && core <= 8) v = (core - 1 == k ? 0x3F80u : 0u) | (core - 1 == k + 1 ? 0x3F800000u : 0u);
        }
        *reinterpret_cast<uint32_t*>(smem + Wd::ones_off + i * 4) = v;
    }
    fence_proxy_async_smem();
    if (warp == kMmaWarp) tmem_alloc(smem_u32(smem + Wd::tmem_off), 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *reinterpret_cast<const volatile uint32_t*>(smem + Wd::tmem_off) + 256u * (uint32_t)team_id;
    unsigned char* ring = smem + (uint32_t)(team_id * R) * Wd::slot;
    const uint32_t w_smem = smem_u32(smem + Wd::w_off);
    bool ok = true;

    if (warp == kWeightWarp) {
        // ---- weights: once, or a pass over them per round -----------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            grid_dependency_wait();
            const unsigned char* src = P.weights + (size_t)h * Wd::weights;
            if constexpr (Wd::resident) {
                mbar_expect_tx(wbar(kWFull), Wd::weights);
                bulk_load_1d(w_smem, src, Wd::weights, wbar(kWFull));
            } else {
                int ws = 0;
                uint32_t phase = 1;
                for (int r = 0; ok && r < rounds; ++r) {
                    const unsigned char* at = src;
                    for (int side = 0; ok && side < 2; ++side)
                        for (int dx = 0; ok && dx < K; ++dx)
                            for (int left = K; left > 0;) {
                                const int g = side ? (left < GV ? left : GV) : (left < GK ? left : GK);
                                left -= g;
                                if (!mbar_wait(wbar(kWEmpty + ws), phase)) { ok = false; break; }
                                mbar_expect_tx(wbar(kWFull + ws), (uint32_t)g * Wd::tap);
                                bulk_load_1d(w_smem + (uint32_t)ws * Wd::chunk, at, (uint32_t)g * Wd::tap, wbar(kWFull + ws));
                                at += (uint32_t)g * Wd::tap;
                                if (++ws == 3) { ws = 0; phase ^= 1u; }
                            }
                }
            }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else if (warp >= kTmaWarp) {
        // ---- TMA thread of a team: K, then V tiles of every block ---------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            int slot = 0;
            uint32_t phase = 1;
            TileWalk at(P.tiles_x, P.tiles_y, 2 * first, 2 * step);
            for (int bi = 0; ok && bi < my_blocks; ++bi, at.next())
                for (int v = 0; v < 2; ++v) {
                    if (!mbar_wait(bar(kEmpty + slot), phase)) { ok = false; break; }
                    mbar_expect_tx(bar(kFull + slot), Wd::slot);
                    const CUtensorMap* map = v ? &map_v : &map_k;
                    const uint32_t dst = smem_u32(ring) + (uint32_t)slot * Wd::slot;
                    // the second tile may be past the last: its image does not exist and it reads as zero
                    int x = at.x + 1, y = at.y, b = at.b;
                    if (x == at.tx) { x = 0; if (++y == at.ty) { y = 0; ++b; } }
                    tma_load_4d(dst, map, bar(kFull + slot), h * kHeadDim, 8 * at.x - Wd::R, 8 * at.y - Wd::R, at.b);
                    tma_load_4d(dst + Wd::plane, map, bar(kFull + slot), h * kHeadDim, 8 * x - Wd::R, 8 * y - Wd::R, b);
                    if (++slot == R) { slot = 0; phase ^= 1u; }
                }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else if (warp >= kMmaWarp) {
        // ---- MMA thread of a team ---------------------------------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            constexpr uint32_t id_l = umma_idesc_bf16(128, N), id16 = umma_idesc_bf16(128, 16), id32 = umma_idesc_bf16(128, 32);
            const uint32_t ones = smem_u32(smem + Wd::ones_off), unit = smem_u32(smem + Wd::unit_off);
            if (Wd::resident && my_blocks > 0) ok = mbar_wait(wbar(kWFull), 0);
            int ws = 0, pb = 0, db = 0;
            uint32_t wphase = 0, pphase = 0, dphase = 1;
            // the next group of weights; `at`: where it is when they are resident
            auto weights = [&](uint32_t at) -> uint32_t {
                if constexpr (Wd::resident) return w_smem + at;
                if (!mbar_wait(wbar(kWFull + ws), wphase)) ok = false;
                return w_smem + (uint32_t)ws * Wd::chunk;
            };
            auto weights_done = [&](bool used) {
                if constexpr (!Wd::resident) {
                    if (used) umma_commit(wbar(kWEmpty + ws)); else mbar_arrive(wbar(kWEmpty + ws));
                    if (++ws == 3) { ws = 0; wphase ^= 1u; }
                }
            };
            for (int r = 0; ok && r < (Wd::resident ? my_blocks : rounds); ++r) {
                if (r >= my_blocks) {                                    // a round without a block of this team
                    for (int i = 0; ok && i < K * (NGK + NGV); ++i) { weights(0); weights_done(false); }
                    continue;
                }
                for (int dx = 0; ok && dx < K; ++dx) {
#pragma unroll
                    for (int gi = 0; gi < NGK; ++gi) {
                        constexpr int GL = K - (NGK - 1) * GK;
                        const int G = gi == NGK - 1 ? GL : GK;
                        const uint32_t w = weights((uint32_t)(dx * K + gi * GK) * Wd::tap);
                        if (!ok || !mbar_wait(bar(kPFull + pb), pphase)) { ok = false; break; }
                        tc_fence_after_sync();
#pragma unroll
                        for (int i = 0; i < G; ++i) {
                            const int t = (gi * GK + i) * K + dx;
                            const uint32_t a = tmem + (uint32_t)(pb * 16 * GK + 16 * i);
                            const uint64_t b = umma_smem_desc(w + i * Wd::tap, N * 16, 128);
                            umma_bf16_ts(tmem + kColL, a, b, id_l, (dx | gi | i) != 0 ? 1u : 0u);
                            umma_bf16_ts(tmem + kColL, a + 8, b + 2 * N, id_l, 1);                    // the other 16 channels
                            const uint64_t one = umma_smem_desc(ones + (uint32_t)(15 - (t & 15)) * 16u, 512, 128);
                            umma_bf16_ts(tmem + kColL + (t & ~15), a, one, id16, 1);
                            umma_bf16_ts(tmem + kColL + (t & ~15), a + 8, one, id16, 1);
                        }
                        umma_commit(bar(kPFree + pb));
                        weights_done(true);
                        if (++pb == PB) { pb = 0; pphase ^= 1u; }
                    }
                }
                if (!ok) break;
                umma_commit(bar(kLFull));
                if (!mbar_wait(bar(kAFull), (uint32_t)r & 1u)) { ok = false; break; }
                for (int dx = 0; ok && dx < K; ++dx) {
#pragma unroll
                    for (int gi = 0; gi < NGV; ++gi) {
                        constexpr int GL = K - (NGV - 1) * GV;
                        const int G = gi == NGV - 1 ? GL : GV;
                        const uint32_t w = weights((uint32_t)(Wd::K2 + dx * K + gi * GV) * Wd::tap);
                        if (!ok || !mbar_wait(bar(kDFree + db), dphase)) { ok = false; break; }
                        tc_fence_after_sync();
                        const uint32_t d = tmem + (uint32_t)(db * 32 * GV);
                        const uint64_t b = umma_smem_desc(w, 128, 2 * KS * 128);
#pragma unroll
                        for (int j = 0; j < KS; ++j) umma_bf16_ts(d, tmem + kColL + 16 * j, b + 16 * j, umma_idesc_bf16(128, 32 * G), j != 0 ? 1u : 0u);
#pragma unroll
                        for (int i = 0; i < G; ++i) {
                            const int t = (gi * GV + i) * K + dx, j = t & 15;
                            // [ones in k = j | zeros] or [zeros | ones in k = j - 8] of the table
                            const uint64_t one = j < 8 ? umma_smem_desc(unit + (uint32_t)(1 + j) * 128u, (uint32_t)(8 - j) * 128u, 1280)
                                                       : umma_smem_desc(unit, (uint32_t)(j - 7) * 128u, 1280);
                            umma_bf16_ts(d + 32 * i, tmem + kColL + (t & ~15), one, id32, 1);
                            umma_bf16_ts(d + 32 * i, tmem + kColL + (t & ~15) + 8, one, id32, 1);
                        }
                        umma_commit(bar(kDFull + db));
                        weights_done(true);
                        if (++db == DB) { db = 0; dphase ^= 1u; }
                    }
                }
            }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else {
        const int wq = warp & 3, half = (warp % kTeamWarps) >> 2, g = lane >> 2, tig = lane & 3;
        const uint32_t quad = tmem + ((uint32_t)(32 * wq) << 16), mine = quad + ((uint32_t)(16 * half) << 16);
        const int C = P.heads * kHeadDim, row0 = 4 * (wq & 1) + 2 * half;
        const size_t row_pitch = (size_t)P.W * C;
        const uint32_t lane_off = (uint32_t)(wq >> 1) * Wd::plane + (uint32_t)(row0 * HP + g) * 64u + (uint32_t)tig * 16u;
        TileWalk walk(P.tiles_x, P.tiles_y, 2 * first + (wq >> 1), 2 * step);
        struct Place { size_t at; bool in[2]; };
        auto place = [&](int bi) {
            Place p;
            const int y = 8 * walk.y + row0, x = 8 * walk.x + g;
            const bool in = 2 * (first + bi * step) + (wq >> 1) < P.tiles && x < P.W;
            p.in[0] = in && y < P.H; p.in[1] = in && y + 1 < P.H;
            p.at = (((size_t)walk.b * P.H + y) * P.W + x) * C + h * kHeadDim + tig * 8;
            return p;
        };
        auto load_q = [&](const Place& p, uint4 (&x)[2]) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                x[r] = make_uint4(0u, 0u, 0u, 0u);
                if (p.in[r]) x[r] = __ldg(reinterpret_cast<const uint4*>(P.q + p.at + r * row_pitch));
            }
        };
        int slot = 0, pb = 0, db = 0;
        uint32_t phase = 0, pphase = 1, dphase = 0;
        const uint32_t zero = (uint32_t)(P.H >> 31);
        float* inv = reinterpret_cast<float*>(smem + Wd::inv_off) + 128 * team_id + 32 * wq;      // of the quadrant's pixels
        auto release = [&]() {
            __syncwarp();
            mbar_arrive_lane0(bar(kEmpty + slot), lane);
            if (++slot == R) { slot = 0; phase ^= 1u; }
        };
        auto release_after = [&](float a, float b) {                // the sums a and b hold what was read from it
            __syncwarp();
            mbar_arrive_lane0_after(bar(kEmpty + slot), lane, a, b, zero);
            if (++slot == R) { slot = 0; phase ^= 1u; }
        };
        Place cur = place(0);
        uint4 x[2];
        if (my_blocks > 0) load_q(cur, x);
        for (int bi = 0; ok && bi < my_blocks; ++bi) {
            // ---- products -------------------------------------------------------------------------------
            if (!warp_wait(bar(kFull + slot), phase)) { ok = false; break; }
            {
                const unsigned char* src = ring + (uint32_t)slot * Wd::slot + lane_off;
#pragma unroll 1
                for (int dx = 0; ok && dx < K; ++dx, src += 64) {
#pragma unroll
                    for (int gi = 0; gi < NGK; ++gi) {
                        constexpr int GL = K - (NGK - 1) * GK;
                        if (!warp_wait(bar(kPFree + pb), pphase)) { ok = false; break; }
                        tc_fence_after_sync();
                        const uint32_t t = mine + (uint32_t)(pb * 16 * GK);
                        if (gi == NGK - 1) store_products<GL, HP>(t, src + gi * GK * HP * 64, x);
                        else store_products<GK, HP>(t, src + gi * GK * HP * 64, x);
                        tmem_wait_st();
                        tc_fence_before_sync();
                        __syncwarp();
                        mbar_arrive_lane0(bar(kPFull + pb), lane);
                        if (++pb == PB) { pb = 0; pphase ^= 1u; }
                    }
                }
            }
            if (!ok) break;
            release();
            const Place out = cur;
            if (bi + 1 < my_blocks) { walk.next(); cur = place(bi + 1); load_q(cur, x); }

            // ---- softmax: thread = pixel of the quadrant; the two warps of a quadrant take turns ----------------
            if (half == (bi & 1)) {
                if (!warp_wait(bar(kLFull), (uint32_t)bi & 1u)) { ok = false; break; }
                tc_fence_after_sync();
                inv[lane] = softmax_in_place<K>(quad + kColL, s_bias, P.scale_log2e);
                tc_fence_before_sync();
                __syncwarp();
                mbar_arrive_lane0(bar(kAFull), lane);
            }

            // ---- values -----------------------------------------------------------------------------------
            float acc[2][8];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[r][c] = 0.f;
            if (!warp_wait(bar(kFull + slot), phase)) { ok = false; break; }
            {
                const unsigned char* src = ring + (uint32_t)slot * Wd::slot + lane_off;
#pragma unroll 1
                for (int dx = 0; ok && dx < K; ++dx, src += 64) {
#pragma unroll
                    for (int gi = 0; gi < NGV; ++gi) {
                        constexpr int GL = K - (NGV - 1) * GV;
                        if (!warp_wait(bar(kDFull + db), dphase)) { ok = false; break; }
                        tc_fence_after_sync();
                        const uint32_t t = mine + (uint32_t)(db * 32 * GV);
                        if (gi == NGV - 1) sum_group<GL, HP>(t, src + gi * GV * HP * 64, acc);
                        else sum_group<GV, HP>(t, src + gi * GV * HP * 64, acc);
                        tc_fence_before_sync();
                        __syncwarp();
                        mbar_arrive_lane0(bar(kDFree + db), lane);
                        if (++db == DB) { db = 0; dphase ^= 1u; }
                    }
                }
            }
            if (!ok) break;
            release_after(acc[0][0], acc[1][0]);
            if (!warp_wait(bar(kAFull), (uint32_t)bi & 1u)) { ok = false; break; }        // long complete: orders the reads of inv
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (out.in[r]) {
                    const float s = inv[16 * half + 8 * r + g];
                    *reinterpret_cast<uint4*>(P.out + out.at + r * row_pitch) =
                        make_uint4(pack_bf16(acc[r][0] * s, acc[r][1] * s), pack_bf16(acc[r][2] * s, acc[r][3] * s),
                                   pack_bf16(acc[r][4] * s, acc[r][5] * s), pack_bf16(acc[r][6] * s, acc[r][7] * s));
                }
        }
        if (!ok && lane == 0) atomicExch(P.status, 1);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(*reinterpret_cast<const volatile uint32_t*>(smem + Wd::tmem_off), 512);
    }
}

template <int K>
cudaError_t launch_prep_t(const Problem& p, void* workspace, cudaStream_t stream) {
    return launch_chained(mma_wide_prep_kernel<K>, dim3((unsigned)((2 * Wide<K>::K2 * 4 * Wide<K>::N + 255) / 256), (unsigned)p.heads), 256, 0, stream, p.wk, p.wv,
                          static_cast<unsigned char*>(workspace));
}

template <int K>
cudaError_t launch_t(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream) {
    using Wd = Wide<K>;
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(mma_wide_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Wd::total);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured[dev] = true;
    }
    WideParams P;
    P.weights = static_cast<const unsigned char*>(workspace);
    P.q = static_cast<const __nv_bfloat16*>(p.q); P.bias = p.bias; P.out = static_cast<__nv_bfloat16*>(p.out); P.status = d_status;
    P.H = p.H; P.W = p.W; P.heads = p.heads;
    P.tiles_x = (p.W + 7) / 8; P.tiles_y = (p.H + 7) / 8;
    const long long tiles = (long long)P.tiles_x * P.tiles_y * p.B;
    if (tiles > 0x3fffffffLL) return cudaErrorInvalidConfiguration;
    P.tiles = (int)tiles;
    P.scale_log2e = kLog2e / sqrtf((float)kHeadDim);
    const int C = p.heads * kHeadDim;
    CUtensorMap mk, mv;
    if (!make_tile_map(&mk, p.k, 2, p.B, p.H, p.W, C, kHeadDim, Wd::HP, Wd::HP) ||
        !make_tile_map(&mv, p.v, 2, p.B, p.H, p.W, C, kHeadDim, Wd::HP, Wd::HP))
        return cudaErrorInvalidValue;
    const long long blocks = (tiles + 1) / 2;
    long long per_head = num_sms / p.heads;
    if (per_head > blocks) per_head = blocks;
    if (per_head < 1) per_head = 1;
    return launch_chained(mma_wide_kernel<K>, dim3((unsigned)(per_head * p.heads)), kThreads, Wd::total, stream, mk, mv, P);
}

}  // namespace

bool mma_wide_supports(slide_attn_dtype dtype, int head_dim, int ksize) {
    return dtype == SLIDE_ATTN_BF16 && head_dim == kHeadDim && (ksize == 3 || ksize == 5 || ksize == 7 || ksize == 9) &&
           tensor_map_available();
}

size_t mma_wide_workspace_bytes(int heads, int ksize) {
    switch (ksize) {
        case 3: return (size_t)heads * Wide<3>::weights;
        case 5: return (size_t)heads * Wide<5>::weights;
        case 7: return (size_t)heads * Wide<7>::weights;
        case 9: return (size_t)heads * Wide<9>::weights;
        default: return 0;
    }
}

// Weights -> images in the order of their use, in `workspace`.
cudaError_t launch_mma_wide_prep(const Problem& p, void* workspace, cudaStream_t stream) {
    switch (p.ksize) {
        case 3: return launch_prep_t<3>(p, workspace, stream);
        case 5: return launch_prep_t<5>(p, workspace, stream);
        case 7: return launch_prep_t<7>(p, workspace, stream);
        case 9: return launch_prep_t<9>(p, workspace, stream);
        default: return cudaErrorInvalidConfiguration;
    }
}

cudaError_t launch_mma_wide(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream) {
    switch (p.ksize) {
        case 3: return launch_t<3>(p, workspace, d_status, num_sms, stream);
        case 5: return launch_t<5>(p, workspace, d_status, num_sms, stream);
        case 7: return launch_t<7>(p, workspace, d_status, num_sms, stream);
        case 9: return launch_t<9>(p, workspace, d_status, num_sms, stream);
        default: return cudaErrorInvalidConfiguration;
    }
}

}  // namespace slide_attn
