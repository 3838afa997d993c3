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
// k = 3; for k >= 7 (400 KB, 1 MB) they are streamed from L2 through a ring that both teams read, 256 pixels per pass over them.
// k = 5 (102 KB, resident) has a kernel of its own below.
//
// Tensor-memory columns of a team (256): logits, later e (chunk of 16 slots: 8 columns e_hi, 8 e_lo, where its logits were), in
// the last N; below them the product groups, later the A' groups.  A group = up to GK (GV) taps of one tap column.
//
// A call: 2 x 128 x 128, 3 heads, k = 7: 137 us with mma.sync, 60 here (issue slots 39 %, tensor pipe 40 %: three rounds for 2.6 blocks
// per team).
#include <type_traits>

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

// What the window makes of a head's weights and of a tile, in every kernel here.
template <int K>
struct Window {
    static constexpr int K2 = K * K, R = K / 2;
    static constexpr int KS = (K2 + 15) / 16;            // K steps of the value side
    static constexpr int N = 16 * KS;                    // columns of the logits
    static constexpr int HP = 8 + 2 * R;                 // edge of a tile with its halo
    static constexpr uint32_t plane = (uint32_t)(HP * HP * 64), slot = 2 * plane;
    static constexpr uint32_t tap = (uint32_t)(N * 64);  // weights of a tap, either side
    static constexpr uint32_t weights = 2u * K2 * tap;   // of a head
};

// mma_wide_kernel: k = 3, 7, 9.
template <int K>
struct Wide : Window<K> {
    using Window<K>::N; using Window<K>::tap; using Window<K>::weights; using Window<K>::slot;
    static constexpr bool resident = K == 3;
    static constexpr int GK = K == 7 ? 4 : 3, GV = K == 9 ? 2 : 3;
    static constexpr int NGK = (K + GK - 1) / GK, NGV = (K + GV - 1) / GV;
    static constexpr int PB = least(3, (256 - N) / (16 * GK)), DB = 2;
    static_assert(DB * 32 * GV <= 256 - N && PB >= 2, "tensor memory");
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
    const unsigned char* weights;    // [head][Window::weights]
    const __nv_bfloat16* q;
    const float* bias;
    __nv_bfloat16* out;
    int* status;
    int H, W, heads;
    int tiles_x, tiles_y, tiles;
    float scale_log2e;
};

constexpr int kPrepThreads = 512;

// Prep: fp32 [C][slot][tap] -> bf16, taps in the order o = dx K + dy (tap t = dy K + dx), first the key side, then the value side; of a
// tap, items of 16 bytes:
//   key tap, item (j, n): k 8j .. 8j + 7 (channels in the order tcgen05.st lays the products out), column n = slot
//   value tap, item (n, j): column n (channel in the order tcgen05.ld hands them out), k 8j .. 8j + 7 = slots
// A block takes eight channels (four of its side) x 16 slots, whose weights are runs of memory, through shared memory to all of their taps.
// Bound by latency: one or two rounds of loads, one of items.  (Before, a thread gathered its eight weights, 4 k^2 bytes apart, from memory: a
// sector for each, which depended on neighbours on the same SM for the rest of it, and when a kernel in front let this one start early its blocks lay on a few
// SMs: forwards of 8 x 56 x 56, 3 heads, k = 3 and then k = 7 58.6 us, here 51.8; 54.7 where nothing starts early.  By themselves, 1 x 14 x 14,
// 8 heads, k = 7 21.5 and 18.3, k = 9 43.2 and 32.4; 4 x 28 x 28, 4 heads, k = 5 9.7 and 9.3; 1 x 14 x 14, 1 head, k = 7 17.4 and 17.7.)
template <int K>
__global__ void __launch_bounds__(kPrepThreads)
mma_wide_prep_kernel(const float* __restrict__ wk, const float* __restrict__ wv, unsigned char* __restrict__ img)
{
    using Wd = Window<K>;
    constexpr int K2 = Wd::K2, Pitch = 16 * K2 + 1;      // odd, so that neither slots nor channels meet in a bank
    __shared__ float s_w[8][Pitch];
    grid_dependency_wait();
    grid_launch_dependents();
    const int side = (int)blockIdx.x / (4 * Wd::KS), four = (int)blockIdx.x % (4 * Wd::KS) / Wd::KS, s0 = 16 * ((int)blockIdx.x % Wd::KS), h = blockIdx.y;
    const int slots = K2 - s0 < 16 ? K2 - s0 : 16;
    {                                                    // two warps a channel
        const int e = threadIdx.x >> 6, i8 = 8 * four + e;
        const int c = side ? 8 * ((i8 & 7) >> 1) + 2 * (i8 >> 3) + (i8 & 1) : 8 * ((i8 & 15) >> 2) + (i8 & 3) + (i8 >= 16 ? 4 : 0);
        const float* src = (side ? wv : wk) + ((size_t)(h * kHeadDim + c) * K2 + s0) * K2;
        constexpr int Deep = 13;                         // loads in flight: one round of them for k <= 7, two for k = 9
        for (int i0 = threadIdx.x & 63; i0 < slots * K2; i0 += 64 * Deep) {
            float x[Deep];
#pragma unroll
            for (int j = 0; j < Deep; ++j) x[j] = i0 + 64 * j < slots * K2 ? __ldg(src + i0 + 64 * j) : 0.f;
#pragma unroll
            for (int j = 0; j < Deep; ++j)
                if (i0 + 64 * j < slots * K2) s_w[e][i0 + 64 * j] = x[j];
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 16 * K2; i += kPrepThreads) {
        const int o = i >> 4, item = i & 15, t = (o % K) * K + o / K;
        float v[8];
        uint32_t at;
        if (side == 0) {
            const int n = s0 + item;
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = n < K2 ? s_w[e][item * K2 + t] - (n == t ? 1.f : 0.f) : 0.f;
            at = (uint32_t)(four * Wd::N * 16 + n * 16);
        } else {
            const int n = item & 7, first = item & 8;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int s = s0 + first + e;
                v[e] = s < K2 ? s_w[n][(first + e) * K2 + t] - (s == t ? 1.f : 0.f) : 0.f;
            }
            at = (uint32_t)(four * (2 * Wd::KS * 128) + (s0 + first) * 16 + n * 16);
        }
        *reinterpret_cast<uint4*>(img + (size_t)h * Wd::weights + (size_t)(side * K2 + o) * Wd::tap + at) =
            make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
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
    using Wd = Window<K>;
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
                // the last commits, here and in the MMA threads, are not on their way any more when the block leaves
                if (ok) ok = wait_last_phases(wbar(kWEmpty), 3, rounds * K * (NGK + NGV));
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
            if (ok) ok = wait_last_phases(bar(kPFree), PB, my_blocks * K * NGK);
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

// ---- k = 5: weights resident, one pipeline over the whole CTA -------------------------------------------------------------------
// The arithmetic above.  As umma_ts_kernel: a warp has a whole quadrant (32 pixels), lane (g, tig) column g and channels 8 tig .. of
// four rows, so that a halo row is read and widened once for up to four of them; the stages have warps of their own.  20 warps: two
// sets of four value warps, which take the blocks in turn, four product, four softmax and four control warps.
// The one-hot part of the value side takes one K step: beside e_hi (K = 25) the softmax leaves, for every tap column, the five e_hi and
// five e_lo of its taps, which meet one table of ones for all columns.  (By a unit column per tap and part, as above, it took 70
// instead of 30 MMAs a block.)
// Tensor memory: a D buffer of 96 columns for the upper three taps of a tap column, two of 64 for the lower two, in turn, two of
// products of 80 (five taps), two tiles of 64: logits in 32 columns, later e_hi in 16 and 8 for each tap column.
//
// Bound by energy when it runs for seconds (1000 W), else by latency: 50.4 M warp instructions at 64 x 56 x 56, 3 heads, in 48 % of the issue
// slots, tensor pipe 42 %, value warps waiting for 60 % of the time.  In two teams of eight warps with two rows each as above 71 M.  Calls, a few
// hundred / for seconds: 64 x 56 x 56, 3 heads 123.5 / 134.5 -> 97 / 112.6 us; 2 x 128 x 128, 3 heads 27.0 -> 24.6.  Without the
// one step for the one-hot part 104.5 / 118.8.
struct Five {
    using Wd = Window<5>;
    static constexpr int K = 5, VSets = 2, KSlots = 2, VSlots = 4, G0 = 3, G1 = 2;
    static constexpr int PWarp = 4 * VSets, SWarp = PWarp + 4, Ctl = SWarp + 4, Threads = (Ctl + 4) * 32;
    static constexpr int LaunchRegs = 96, ValueRegs = 136, ProductRegs = 104, SoftmaxRegs = 64, ControlRegs = 40;      // a thread: at the launch, then
    static_assert(VSets * ValueRegs + ProductRegs + SoftmaxRegs + ControlRegs <= Threads / 128 * LaunchRegs, "registers");
    static constexpr uint32_t ColD = 0, ColD1 = 96, OtherD1 = 96 ^ 160, ColP = 224, OtherP = 224 ^ 304, ColL = 384;       // x ^ Other: the other one of two
    static constexpr uint32_t TapBytes = 5 * 4 * 256;             // table of ones: [tap][four groups of 8 columns][k / 8][column][8 k]
    static constexpr uint32_t v_off = KSlots * Wd::slot, w_off = v_off + VSlots * Wd::slot, ones_off = w_off + Wd::weights, unit_off = ones_off + kOnesBytes,
                              bias_off = unit_off + TapBytes, inv_off = bias_off + 112, bar_off = inv_off + 2 * 128 * 4;
    // Pairs of barriers are told apart by bit 3 of their address.  DFull: [set][tap column][upper, lower]: each has one set of readers, which
    // meets all of its phases.
    enum : int { KFull = 0, KEmpty = KFull + KSlots, VFull = KEmpty + KSlots, VEmpty = VFull + VSlots, PReady = VEmpty + VSlots, PFree = PReady + 2,
                 LFull = PFree + 2, EReady = LFull + 2, EFree = EReady + 2, DFree1 = EFree + 2, DFree = DFree1 + 2, Weights, DFull, Bars = DFull + VSets * K * 2 };
    static_assert(PReady % 2 == 0, "pairs");
    static constexpr uint32_t tmem_off = bar_off + 8 * Bars, total = tmem_off + 16 + 128;
    static_assert(total <= kMaxSmem && VSlots % VSets == 0, "shared memory; a slot of V has one set of readers");
};

__global__ void __launch_bounds__(Five::Threads, 1)
mma_five_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const WideParams P)
{
    using F = Five;
    using Wd = F::Wd;
    constexpr int K = F::K, HP = Wd::HP;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const uint32_t bars = smem_u32(smem + F::bar_off);
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    float* s_bias = reinterpret_cast<float*>(smem + F::bias_off);
    float* s_inv = reinterpret_cast<float*>(smem + F::inv_off);          // [block parity][pixel]: 1 / sum of the weights

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int h = blockIdx.x % P.heads, rank = blockIdx.x / P.heads, nrank = (int)gridDim.x / P.heads;
    const int blocks = (P.tiles + 1) >> 1, my_blocks = rank < blocks ? (blocks - rank + nrank - 1) / nrank : 0;

    if (threadIdx.x < F::Bars) {                                   // a thread a barrier: one after the other they take 0.2 us
        const int i = threadIdx.x;
        auto in = [&](int first, int n) { return i >= first && i < first + n; };
        const bool warps = in(F::KEmpty, F::KSlots) || in(F::VEmpty, F::VSlots) || in(F::PReady, 2) || in(F::EReady, 2) || in(F::DFree1, 3);
        mbar_init_only(bar(i), warps ? 4u : 1u);
        mbar_init_fence();
    }
    for (int i = threadIdx.x; i < Wd::K2; i += F::Threads) s_bias[i] = P.bias ? P.bias[h * Wd::K2 + i] * kLog2e : 0.f;
    for (uint32_t i = threadIdx.x; i < (kOnesBytes + F::TapBytes) / 4; i += F::Threads) {
        uint32_t v = 0;
        if (i < kOnesBytes / 4) {
            if (((i * 4) & 511u) >> 4 == 15) v = kOnesBf16x2;
        } else {                                                  // k = e_hi of tap 0 .. 4, e_lo of tap 0 .. 4; 32 columns a tap
            const uint32_t b = i * 4 - kOnesBytes, tap = b >> 10, k = (b >> 7 & 1u) * 8u + ((b & 15u) >> 1);
            v = (k == tap || k == 5 + tap ? 0x3F80u : 0u) | (k + 1 == tap || k + 1 == 5 + tap ? 0x3F800000u : 0u);
        }
        *reinterpret_cast<uint32_t*>(smem + F::ones_off + i * 4) = v;
    }
    fence_proxy_async_smem();
    if (warp == F::Ctl) tmem_alloc(smem_u32(smem + F::tmem_off), 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *reinterpret_cast<const volatile uint32_t*>(smem + F::tmem_off);
    const int C = P.heads * kHeadDim, g = lane >> 2, tig = lane & 3, q = warp & 3;
    const size_t row_pitch = (size_t)P.W * C;
    const uint32_t lane_off = (uint32_t)(q >> 1) * Wd::plane + (uint32_t)(4 * (q & 1) * HP + g) * 64u + (uint32_t)tig * 16u;
    // the lane's pixel in its first row, and how many of its four rows are inside (tile `i` past the last: none)
    struct Place { size_t at; int rows; };
    auto place = [&](const TileWalk& w, int i) {
        Place p;
        const int y = 8 * w.y + 4 * (q & 1), x = 8 * w.x + g;
        p.rows = i < P.tiles && x < P.W ? P.H - y : 0;
        p.at = (((size_t)w.b * P.H + y) * P.W + x) * C + h * kHeadDim + tig * 8;
        return p;
    };
    bool ok = true;

    if (warp < F::PWarp) {
        // ---- values -----------------------------------------------------------------------------------------
        reg_share<F::ValueRegs, F::LaunchRegs>();
        const int set = warp >> 2;
        const uint32_t tq = tmem + ((uint32_t)(32 * q) << 16);
        TileWalk walk(P.tiles_x, P.tiles_y, 2 * (rank + set * nrank) + (q >> 1), 2 * F::VSets * nrank);
        const uint32_t zero = (uint32_t)(P.H >> 31), ready = bar(F::EReady + set);
        const float* inv = s_inv + 128 * set + 32 * q + g;
        int slot = set;
        uint32_t phase = 0, parity = 0;                            // of the slot; of the block
#pragma unroll 1
        for (int blk = set; blk < my_blocks; blk += F::VSets) {
            const unsigned char* src = smem + F::v_off + (uint32_t)slot * Wd::slot + lane_off;
            wait_or_give_up(bar(F::VFull + slot), phase, ok);
            wait_or_give_up(ready, parity, ok);
            float s[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] = inv[8 * i];
            float acc[4][8];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[i][c] = 0.f;
            uint32_t full = bar(F::DFull + 2 * K * set), free1 = bar(F::DFree1 + set), t1 = tq + (set ? 160u : 96u);        // buffer 5 blk + dx mod 2
#pragma unroll 1
            for (int dx = 0; dx < K; ++dx, src += 64, full += 16u, free1 ^= 8u, t1 ^= F::OtherD1) {
                uint4 y[8];
                float f[8][8];
                auto load = [&](int r) { y[r] = *reinterpret_cast<const uint4*>(src + r * HP * 64); };
                auto widen = [&](int r) {
                    f[r][0] = bf16_lo(y[r].x); f[r][1] = bf16_hi(y[r].x); f[r][2] = bf16_lo(y[r].y); f[r][3] = bf16_hi(y[r].y);
                    f[r][4] = bf16_lo(y[r].z); f[r][5] = bf16_hi(y[r].z); f[r][6] = bf16_lo(y[r].w); f[r][7] = bf16_hi(y[r].w);
                };
                // taps dy0 .. dy0 + G - 1 of the column, pixel rows 2m, 2m + 1: their A' from `t`
                auto ask = [&](auto G, uint32_t t, uint32_t (&d)[3][16]) {
#pragma unroll
                    for (int i = 0; i < decltype(G)::value; ++i) tmem_ld_16x256b_x4_nowait(t + 32 * i, d[i]);
                };
                auto sum = [&](auto G, int dy0, int m, uint32_t (&d)[3][16]) {
#pragma unroll
                    for (int i = 0; i < decltype(G)::value; ++i) {
                        tmem_pass(d[i]);
#pragma unroll
                        for (int r = 0; r < 2; ++r)
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                ffma2(acc[2 * m + r][2 * j], acc[2 * m + r][2 * j + 1], __uint_as_float(d[i][4 * j + 2 * r]), __uint_as_float(d[i][4 * j + 2 * r + 1]),
                                      f[2 * m + r + dy0 + i][2 * j], f[2 * m + r + dy0 + i][2 * j + 1]);
                    }
                };
                using G0 = std::integral_constant<int, F::G0>;
                using G1 = std::integral_constant<int, F::G1>;
                uint32_t d[3][16];
#pragma unroll
                for (int r = 0; r < 6; ++r) load(r);
                wait_or_give_up(full, parity, ok);
                tc_fence_after_sync();
                ask(G0(), tq, d);
                widen(0); widen(1); widen(2); widen(3);
                tmem_wait_ld();
                sum(G0(), 0, 0, d);
                ask(G0(), tq + (16u << 16), d);
                widen(4); widen(5);
                load(6); load(7);
                tmem_wait_ld();
                tc_fence_before_sync();
                mbar_arrive_lane0(bar(F::DFree), lane);
                sum(G0(), 0, 1, d);
                wait_or_give_up(full + 8u, parity, ok);
                tc_fence_after_sync();
                ask(G1(), t1, d);
                widen(6); widen(7);
                tmem_wait_ld();
                sum(G1(), 3, 0, d);
                ask(G1(), t1 + (16u << 16), d);
                tmem_wait_ld();
                tc_fence_before_sync();
                mbar_arrive_lane0(free1, lane);
                sum(G1(), 3, 1, d);
            }
            // row 0 of the accumulators holds what was read last of halo rows 0 - 4, row 3 of 3 - 7
            mbar_arrive_lane0_after(bar(F::VEmpty + slot), lane, acc[0][0], acc[3][0], zero);
            if ((slot += F::VSets) >= F::VSlots) { slot = set; phase ^= 1u; }
            parity ^= 1u;
            const Place out = place(walk, 2 * (rank + blk * nrank) + (q >> 1));
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < out.rows)
                    *reinterpret_cast<uint4*>(P.out + out.at + i * row_pitch) =
                        make_uint4(pack_bf16(acc[i][0] * s[i], acc[i][1] * s[i]), pack_bf16(acc[i][2] * s[i], acc[i][3] * s[i]),
                                   pack_bf16(acc[i][4] * s[i], acc[i][5] * s[i]), pack_bf16(acc[i][6] * s[i], acc[i][7] * s[i]));
            walk.next();
        }
    } else if (warp < F::SWarp) {
        // ---- products ---------------------------------------------------------------------------------------
        reg_share<F::ProductRegs, F::LaunchRegs>();
        uint32_t t = tmem + F::ColP + ((uint32_t)(32 * q) << 16), free = bar(F::PFree), ppar = 1, pb = 0;      // chunk 5 blk + dx: buffer, its barrier, phase
        TileWalk walk(P.tiles_x, P.tiles_y, 2 * rank + (q >> 1), 2 * nrank);
        uint4 x[4], xn[4];                                         // q of this block and of the next
        auto load_q = [&](int blk) {
            const Place p = place(walk, 2 * (rank + blk * nrank) + (q >> 1));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                xn[i] = make_uint4(0u, 0u, 0u, 0u);
                if (i < p.rows) xn[i] = __ldg(reinterpret_cast<const uint4*>(P.q + p.at + i * row_pitch));
            }
        };
        int slot = 0;
        uint32_t phase = 0;
        if (my_blocks > 0) load_q(0);
#pragma unroll 1
        for (int blk = 0; blk < my_blocks; ++blk) {
            const unsigned char* src = smem + (uint32_t)slot * Wd::slot + lane_off;
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = xn[i];
            walk.next();
            if (blk + 1 < my_blocks) load_q(blk + 1);
            wait_or_give_up(bar(F::KFull + slot), phase, ok);
#pragma unroll 1
            for (int dx = 0; dx < K; ++dx, src += 64) {
                uint4 y[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) y[r] = *reinterpret_cast<const uint4*>(src + r * HP * 64);
                wait_or_give_up(free, ppar, ok);
                tc_fence_after_sync();
#pragma unroll
                for (int i = 0; i < K; ++i)
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const uint4 x0 = x[2 * m], x1 = x[2 * m + 1], y0 = y[2 * m + i], y1 = y[2 * m + 1 + i];
                        const uint32_t r[8] = {hmul2_bf16(x0.x, y0.x), hmul2_bf16(x0.y, y0.y), hmul2_bf16(x1.x, y1.x), hmul2_bf16(x1.y, y1.y),
                                               hmul2_bf16(x0.z, y0.z), hmul2_bf16(x0.w, y0.w), hmul2_bf16(x1.z, y1.z), hmul2_bf16(x1.w, y1.w)};
                        tmem_st_16x256b_x2(t + ((uint32_t)(16 * m) << 16) + 16 * i, r);
                    }
                tmem_wait_st();
                tc_fence_before_sync();
                mbar_arrive_lane0(free - 8u * (uint32_t)(F::PFree - F::PReady), lane);
                t ^= F::OtherP; free ^= 8u; ppar ^= pb; pb ^= 1u;
            }
            mbar_arrive_lane0(bar(F::KEmpty + slot), lane);       // the products of what was read are in tensor memory
            if (++slot == F::KSlots) { slot = 0; phase ^= 1u; }
        }
    } else if (warp < F::Ctl) {
        // ---- softmax: thread = pixel ----------------------------------------------------------------------------
        reg_share<F::SoftmaxRegs, F::LaunchRegs>();
        const uint32_t tq = tmem + F::ColL + ((uint32_t)(32 * q) << 16);
#pragma unroll 1
        for (int blk = 0; blk < my_blocks; ++blk) {
            const uint32_t tile = (uint32_t)blk & 1u;
            wait_or_give_up(bar(F::LFull) + 8u * tile, (uint32_t)blk >> 1 & 1u, ok);
            tc_fence_after_sync();
            float l[32];
            tmem_ld_32x32b_x32(tq + 64u * tile, l);
            // the largest of all slots first: a running one is -inf while all slots so far are masked by a bias of -inf
            float m = -INFINITY, z = 0.f;
#pragma unroll
            for (int i = 0; i < Wd::K2; ++i) { l[i] = fmaf(l[i], P.scale_log2e, s_bias[i]); m = fmaxf(m, l[i]); }
            uint32_t hi[16], lo[13];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float e0 = 2 * i < Wd::K2 ? fast_exp2(l[2 * i] - m) : 0.f, e1 = 2 * i + 1 < Wd::K2 ? fast_exp2(l[2 * i + 1] - m) : 0.f;
                z += e0; z += e1;
                hi[i] = i < 13 ? pack_bf16(e0, e1) : 0u;
                if (i < 13) lo[i] = pack_bf16(e0 - bf16_lo(hi[i]), e1 - bf16_hi(hi[i]));
            }
            tmem_st_32x32b_x16(tq + 64u * tile, hi);
            // halves of two words as one
            auto both = [&](const uint32_t (&a)[16], int i, const uint32_t (&b)[16], int j) {
                return __byte_perm(a[i >> 1], b[j >> 1], (i & 1 ? 0x32u : 0x10u) | (j & 1 ? 0x7600u : 0x5400u));
            };
            uint32_t low[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) low[i] = i < 13 ? lo[i] : 0u;
#pragma unroll
            for (int dx = 0; dx < K; ++dx) {
                const uint32_t row[8] = {both(hi, dx, hi, 5 + dx), both(hi, 10 + dx, hi, 15 + dx), both(hi, 20 + dx, low, dx), both(low, 5 + dx, low, 10 + dx),
                                         both(low, 15 + dx, low, 20 + dx), 0u, 0u, 0u};
                tmem_st_32x32b_x8(tq + 64u * tile + 16 + 8 * dx, row);
            }
            tmem_wait_st();
            s_inv[128 * tile + 32 * q + lane] = 1.f / z;
            tc_fence_before_sync();
            __syncwarp();
            mbar_arrive_lane0(bar(F::EReady) + 8u * tile, lane);
        }
    } else {
        reg_share<F::ControlRegs, F::LaunchRegs>();
        // no copy or commit is on its way when the block leaves, whatever its readers have given up on
        auto drain = [&](int first, int slots, int uses) { ok = wait_last_phases(bar(first), slots, uses) && ok; };
        auto load_tiles = [&](uint32_t dst, const CUtensorMap* map, uint32_t full, const TileWalk& at) {
            mbar_expect_tx(full, Wd::slot);
            // the second tile may be past the last: its image does not exist and it reads as zero
            int x = at.x + 1, y = at.y, b = at.b;
            if (x == at.tx) { x = 0; if (++y == at.ty) { y = 0; ++b; } }
            tma_load_4d(dst, map, full, h * kHeadDim, 8 * at.x - Wd::R, 8 * at.y - Wd::R, at.b);
            tma_load_4d(dst + Wd::plane, map, full, h * kHeadDim, 8 * x - Wd::R, 8 * y - Wd::R, b);
        };
        uint32_t leader;
        if (elect_one(leader) && my_blocks > 0) {
            const uint32_t w = smem_u32(smem + F::w_off);
            if (warp == F::Ctl) {
                // ---- key MMAs -------------------------------------------------------------------------------
                constexpr uint32_t id_l = umma_idesc_bf16(128, Wd::N), id16 = umma_idesc_bf16(128, 16);
                // descriptors, lower halves: weights of tap (0, 0); the ones of column 15 in column 15
                const uint64_t wd = umma_smem_desc(w, Wd::N * 16, 128), od = umma_smem_desc(smem_u32(smem + F::ones_off), 512, 128);
                const uint32_t w_lo = (uint32_t)wd, w_hi = (uint32_t)(wd >> 32), o_lo = (uint32_t)od + 15u, o_hi = (uint32_t)(od >> 32);
                uint32_t p = tmem + F::ColP, ready = bar(F::PReady), ppar = 0, pb = 0;
                ok = mbar_wait<true>(bar(F::Weights), 0);
#pragma unroll 1
                for (int blk = 0; ok && blk < my_blocks; ++blk) {
                    const uint32_t tile = (uint32_t)blk & 1u, l = tmem + F::ColL + 64u * tile;
                    if (!mbar_wait<true>(bar(F::EFree) + 8u * tile, ((uint32_t)blk >> 1 & 1u) ^ 1u)) { ok = false; break; }
#pragma unroll 1
                    for (int dx = 0; dx < K; ++dx) {
                        if (!mbar_wait<true>(ready, ppar)) { ok = false; break; }
                        tc_fence_after_sync();
#pragma unroll
                        for (int i = 0; i < K; ++i) {
                            const uint32_t t = (uint32_t)(i * K + dx), a = p + 16 * i;
                            const uint32_t b = w_lo + (uint32_t)dx * (K * Wd::tap / 16) + i * (Wd::tap / 16), one = o_lo - (t & 15u), lt = l + (t & 16u);
                            umma_bf16_ts(l, a, b, w_hi, id_l, i != 0 ? 1u : (uint32_t)dx);
                            umma_bf16_ts(l, a + 8, b + 2 * Wd::N, w_hi, id_l, 1);                     // the other 16 channels
                            umma_bf16_ts(lt, a, one, o_hi, id16, 1);
                            umma_bf16_ts(lt, a + 8, one, o_hi, id16, 1);
                        }
                        umma_commit(ready + 8u * (uint32_t)(F::PFree - F::PReady));
                        p ^= F::OtherP; ready ^= 8u; ppar ^= pb; pb ^= 1u;
                    }
                    if (ok) umma_commit(bar(F::LFull) + 8u * tile);
                }
                if (ok) drain(F::PFree, 2, K * my_blocks);
            } else if (warp == F::Ctl + 1) {
                // ---- value MMAs -----------------------------------------------------------------------------
                const uint64_t wd = umma_smem_desc(w + (uint32_t)Wd::K2 * Wd::tap, 128, 2 * Wd::KS * 128), ud = umma_smem_desc(smem_u32(smem + F::unit_off), 128, 256);
                const uint32_t w_lo = (uint32_t)wd, w_hi = (uint32_t)(wd >> 32), u_lo = (uint32_t)ud, u_hi = (uint32_t)(ud >> 32);
                uint32_t d1 = tmem + F::ColD1, free1 = bar(F::DFree1), dpar = 1, dpar1 = 1, db = 0;
                ok = mbar_wait<true>(bar(F::Weights), 0);
#pragma unroll 1
                for (int blk = 0; ok && blk < my_blocks; ++blk) {
                    const uint32_t tile = (uint32_t)blk & 1u, e = tmem + F::ColL + 64u * tile;
                    if (!mbar_wait<true>(bar(F::EReady) + 8u * tile, (uint32_t)blk >> 1 & 1u)) { ok = false; break; }
                    uint32_t full = bar(F::DFull) + 16u * K * tile;
#pragma unroll 1
                    for (int dx = 0; ok && dx < K; ++dx, full += 16u) {
#pragma unroll
                        for (int gi = 0; gi < 2; ++gi) {
                            const int G = gi ? F::G1 : F::G0;
                            if (!mbar_wait<true>(gi ? free1 : bar(F::DFree), gi ? dpar1 : dpar)) { ok = false; break; }
                            tc_fence_after_sync();
                            const uint32_t d = gi ? d1 : tmem + F::ColD;
                            const uint32_t b = w_lo + (uint32_t)dx * (K * Wd::tap / 16) + gi * (F::G0 * Wd::tap / 16);
#pragma unroll
                            for (int j = 0; j < Wd::KS; ++j) umma_bf16_ts(d, e + 8 * j, b + 16 * j, w_hi, umma_idesc_bf16(128, 32 * G), j != 0 ? 1u : 0u);
                            umma_bf16_ts(d, e + 16 + 8u * (uint32_t)dx, u_lo + gi * (F::G0 * 64), u_hi, umma_idesc_bf16(128, 32 * G), 1);
                            umma_commit(full + 8u * gi);
                        }
                        d1 ^= F::OtherD1; free1 ^= 8u; dpar ^= 1u; dpar1 ^= db; db ^= 1u;
                    }
                    if (ok) umma_commit(bar(F::EFree) + 8u * tile);
                }
                if (ok) drain(F::EFree, 2, my_blocks);
            } else {
                // ---- the head's weights and K, or V -------------------------------------------------------------
                const bool v = warp == F::Ctl + 3;
                if (!v) {
                    grid_dependency_wait();
                    mbar_expect_tx(bar(F::Weights), Wd::weights);
                    bulk_load_1d(w, P.weights + (size_t)h * Wd::weights, Wd::weights, bar(F::Weights));
                }
                const int slots = v ? F::VSlots : F::KSlots, full = v ? F::VFull : F::KFull, empty = v ? F::VEmpty : F::KEmpty;
                const uint32_t ring = smem_u32(smem) + (v ? F::v_off : 0u);
                TileWalk at(P.tiles_x, P.tiles_y, 2 * rank, 2 * nrank);
                int slot = 0, blk = 0;
                uint32_t phase = 1;
#pragma unroll 1
                for (; blk < my_blocks; ++blk, at.next()) {
                    if (!mbar_wait<true>(bar(empty + slot), phase)) { ok = false; break; }
                    load_tiles(ring + (uint32_t)slot * Wd::slot, v ? &map_v : &map_k, bar(full + slot), at);
                    if (++slot == slots) { slot = 0; phase ^= 1u; }
                }
                drain(full, slots, blk);
                if (!v) ok = mbar_wait<true>(bar(F::Weights), 0) && ok;
            }
        }
        __syncwarp();
    }
    if (!ok) atomicExch(P.status, 1);
    tc_fence_before_sync();
    __syncthreads();
    if (warp == F::Ctl) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
}

template <int K>
cudaError_t launch_prep_t(const Problem& p, void* workspace, cudaStream_t stream) {
    return launch_chained(mma_wide_prep_kernel<K>, dim3((unsigned)(8 * Window<K>::KS), (unsigned)p.heads), kPrepThreads, 0, stream, p.wk, p.wv,
                          static_cast<unsigned char*>(workspace));
}

template <int K>
cudaError_t launch_t(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream) {
    using Wd = Window<K>;
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !configured[dev]) {
        if constexpr (K == 5) e = cudaFuncSetAttribute(mma_five_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Five::total);
        else e = cudaFuncSetAttribute(mma_wide_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Wide<K>::total);
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
    const dim3 grid((unsigned)(per_head * p.heads));
    if constexpr (K == 5) return launch_chained(mma_five_kernel, grid, Five::Threads, Five::total, stream, mk, mv, P);
    else return launch_chained(mma_wide_kernel<K>, grid, kThreads, Wide<K>::total, stream, mk, mv, P);
}

}  // namespace

bool mma_wide_supports(slide_attn_dtype dtype, int head_dim, int ksize) {
    return dtype == SLIDE_ATTN_BF16 && head_dim == kHeadDim && (ksize == 3 || ksize == 5 || ksize == 7 || ksize == 9) &&
           tensor_map_available();
}

size_t mma_wide_workspace_bytes(int heads, int ksize) {
    switch (ksize) {
        case 3: return (size_t)heads * Window<3>::weights;
        case 5: return (size_t)heads * Window<5>::weights;
        case 7: return (size_t)heads * Window<7>::weights;
        case 9: return (size_t)heads * Window<9>::weights;
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
