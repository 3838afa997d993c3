// Projections of a Slide-Attention block (Eq. 1: q = x W_q, k = x W_k, v = x W_v; Eq. 3: Concat(heads) W_o)
// as one persistent tcgen05 GEMM:  Y[rows x N] = X[rows x K] W[K x N], X and Y bf16 (token-major, channels
// contiguous), W given in fp32 and rounded to bf16 once as each CTA lays it out in its shared memory, fp32
// accumulation in tensor memory.  One launch per projection call.
//
// The operand X goes registers -> tensor memory and the result tensor memory -> registers, both in the 16x256b
// shape, whose lane (g, tig) has rows g and g + 8 of a warp's 16.  The orders of K and of the columns of W are free, so W is
// laid out such that a lane's share of a UNIT of U channels (32, or 16 where the channels are not a multiple of 32) is
// U / 4 consecutive channels: X is read and Y written as one 16-byte (8-byte) access per row and unit, four lanes to 64
// (32) contiguous bytes, with no shared memory in between, and all shared memory is left to W.
//
// Warps: 0-7 load X (16 rows of a 128-row tile each, up to three tiles in registers ahead of their place in tensor memory),
// 8-15 write Y (16 rows of each accumulator of up to 64 columns: a CHUNK), 16 the MMA thread.  Tensor memory: tiles of X in
// columns 0-255, four accumulators above.  Every wait is bounded; a wait that runs out sets the status word and the kernel
// still releases tensor memory.
//
// Columns are split over `groups` of CTAs: CTA c has group c mod groups and the tiles of rank c / groups, in steps.  A CTA moves
// its weights once and 256 (K + cols) bytes per tile; the group count that makes this least for the CTA with the most tiles is
// taken.  It is 1 for long inputs whose W fits shared memory, and grows where there are fewer tiles than SMs or W does not fit.
//
// W comes as the image that proj_prep_kernel wrote, where the caller has room for one, otherwise every CTA lays its columns out
// itself (proj_wants_image).
//
// Bound by memory traffic (X once per group, Y) where the input is long, by the start of a CTA (tensor memory, weights, first
// tile: 3 us) where it is short.  Before, X came by TMA as boxes of 8 channels (a 16-byte row a cycle), the result went through
// shared memory, and what that left for W made a 256-channel block eleven launches, each CTA laying W out from fp32.  A block
// call, before and here: 64 x 56 x 56 x 2 heads of 32 66.0 and 59.0 us (Eq. 1 22, Eq. 3 13.3 of it), 30 x 28 x 42 x 6
// 68.4 and 43.2, 8 x 115 x 70 x 8 244 and 92.2 (Eq. 1 31.5: 4.2 TB/s), 1 x 14 x 14 x 8 89.8 and 14.7 us.
// Not kept: loads and stores by the same warps in two teams (the loads' latency was exposed: 63.0 / 99.7 us for 2 and 3 heads
// against 59.0 / 89.8), two sets of store warps with fewer tiles in flight (62.7 / 90.1).
#include "common.cuh"
#include "ptx.cuh"

namespace slide_attn {

namespace {

constexpr int kLoadWarps = 8, kStoreWarps = 8, kMmaWarp = kLoadWarps + kStoreWarps;
constexpr int kThreads = (kMmaWarp + 1) * 32;
constexpr int kChunk = 64;                                       // columns of an accumulator
constexpr uint32_t kColD = 256;                                  // X in the columns below
constexpr int kMaxX = 4, kAccs = 4;                              // tiles of X in tensor memory, accumulators
constexpr uint32_t kMaxSmem = 227 * 1024;
enum : int { kXFull = 0, kXFree = kXFull + kMaxX, kDFull = kXFree + kMaxX, kDFree = kDFull + kAccs, kWeights = kDFree + kAccs, kBars };
constexpr uint32_t kMisc = 8 * kBars + 16 + 128;                 // barriers, the address of tensor memory, alignment

struct ProjParams {
    const __nv_bfloat16* x;      // [rows][K]
    const float* w;              // nmat row-major [K][ycols] matrices, one after the other
    const unsigned char* image;  // the same as proj_prep_kernel lays it out, or null
    __nv_bfloat16* y[3];         // output tensors, each [rows][ycols]
    int ycols;                   // channels of one output tensor = columns of one weight matrix
    int rows, K;
    int groups, units, per_group; // units of U columns: in all, of a group (the last one may have fewer)
    int* status;
    bool early;                   // let the kernel behind this one start before this one is complete
};

// channel of K index / column n within a unit: the order in which tcgen05.st lays X out, and in which tcgen05.ld hands Y out
template <int U> __device__ __forceinline__ int channel_of_k(int k) { return U == 32 ? 8 * ((k & 15) >> 2) + (k & 3) + (k >= 16 ? 4 : 0) : k; }
template <int U> __device__ __forceinline__ int channel_of_n(int n) { return (U / 4) * ((n & 7) >> 1) + 2 * (n >> 3) + (n & 1); }

template <int U> struct Piece;                                   // a lane's channels of a unit
template <> struct Piece<32> { using type = uint4; };
template <> struct Piece<16> { using type = uint2; };

__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}
__device__ __forceinline__ void store_x(uint32_t t, const uint4& a, const uint4& b) {
    const uint32_t r[8] = {a.x, a.y, b.x, b.y, a.z, a.w, b.z, b.w};
    tmem_st_16x256b_x2(t, r);
}
__device__ __forceinline__ void store_x(uint32_t t, const uint2& a, const uint2& b) {
    const uint32_t r[4] = {a.x, a.y, b.x, b.y};
    tmem_st_16x256b_x1(t, r);
}
__device__ __forceinline__ uint32_t pack_bits(uint32_t a, uint32_t b) { return pack_bf16(__uint_as_float(a), __uint_as_float(b)); }

// Image of the weights: [8 columns][K / 8][column][8 k] bf16, columns and k of a unit in the orders above; the columns of
// a group are one piece of it.  Item i of `cols` columns from `col` on: 16 bytes; 32 or 16 consecutive items take the columns of a
// unit, so that their fp32 reads are whole lines.
template <int U>
__device__ __forceinline__ void build_item(const float* __restrict__ w, int K, int ycols, int col, int cols, unsigned char* img, int i) {
    const int kg = i / cols, nl = i - kg * cols, n = nl % U, unit_col = col + nl - n, mat = unit_col / ycols;
    const float* src = w + (size_t)mat * K * ycols + (unit_col - mat * ycols + channel_of_n<U>(n));
    const int k0 = kg * 8 / U * U, kin = kg * 8 % U;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = src[(size_t)(k0 + channel_of_k<U>(kin + e)) * ycols];
    *reinterpret_cast<uint4*>(img + (size_t)(nl >> 3) * K * 16 + kg * 128 + (nl & 7) * 16) =
        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}

// The images of two sets of matrices at once (a block's: Eq. 1 and Eq. 3).
template <int U>
__global__ void __launch_bounds__(256)
proj_prep_kernel(const float* __restrict__ wa, int cols_a, unsigned char* __restrict__ image_a, const float* __restrict__ wb, int cols_b,
                 unsigned char* __restrict__ image_b, int K, int ycols)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const int i = (int)(blockIdx.x * 256 + threadIdx.x), items_a = cols_a * (K >> 3), items_b = cols_b * (K >> 3);
    if (i < items_a) build_item<U>(wa, K, ycols, 0, cols_a, image_a, i);
    else if (i - items_a < items_b) build_item<U>(wb, K, ycols, 0, cols_b, image_b, i - items_a);
}

// U: channels of a unit; NS: K rounded up to 64, in 64s.
template <int U, int NS>
__global__ void __launch_bounds__(kThreads, 1)
proj_kernel(const ProjParams P)
{
    using Pc = typename Piece<U>::type;
    constexpr int XU = NS * 64 / U, CU = kChunk / U;             // units of X, of a chunk
    constexpr int TD = NS == 1 ? 3 : NS == 2 ? 2 : 1;            // tiles of X in registers
    constexpr int XB = NS == 1 ? 4 : NS == 2 ? 4 : 2;            // and in tensor memory, 32 NS columns each
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int group = (int)blockIdx.x % P.groups, rank = (int)blockIdx.x / P.groups, nrank = (int)gridDim.x / P.groups;
    const int unit0 = group * P.per_group, units = P.units - unit0 < P.per_group ? P.units - unit0 : P.per_group;
    const int ncols = units * U, nchunks = (ncols + kChunk - 1) / kChunk;
    const int ntiles = (P.rows + 127) >> 7, my_tiles = rank < ntiles ? (ntiles - rank + nrank - 1) / nrank : 0;
    const uint32_t w_bytes = (uint32_t)P.per_group * U * (uint32_t)P.K * 2u;     // of the widest group; a multiple of 512
    const uint32_t bars = smem_u32(smem) + w_bytes;
    unsigned char* tmem_slot = smem + w_bytes + 8u * kBars;
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };

    if (threadIdx.x == 0) {
        for (int i = 0; i < kMaxX; ++i) { mbar_init_only(bar(kXFull + i), kLoadWarps); mbar_init_only(bar(kXFree + i), 1); }
        for (int i = 0; i < kAccs; ++i) { mbar_init_only(bar(kDFull + i), 1); mbar_init_only(bar(kDFree + i), kStoreWarps); }
        mbar_init_only(bar(kWeights), P.image ? 1 : kMmaWarp);
        mbar_init_fence();
    }
    if (warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *reinterpret_cast<const volatile uint32_t*>(tmem_slot);
    // The kernel may have been launched before the kernels ahead of it in the stream completed.
    grid_dependency_wait();
    bool ok = true;
    auto build = [&]() {                                         // this group's weights by the other warps
        if (P.image) return;
        const int items = ncols * (P.K >> 3);
#pragma unroll 2
        for (int i = (int)threadIdx.x; i < items; i += kMmaWarp * 32) build_item<U>(P.w, P.K, P.ycols, unit0 * U, ncols, smem, i);
        fence_proxy_async_smem();                // the tensor core reads these bytes through the async proxy
        __syncwarp();
        mbar_arrive_lane0(bar(kWeights), lane);
    };

    if (warp == kMmaWarp) {
        // ---- MMA thread -----------------------------------------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            const uint32_t w_smem = smem_u32(smem);
            if (P.image) {
                mbar_expect_tx(bar(kWeights), (uint32_t)ncols * (uint32_t)P.K * 2u);
                bulk_load_1d(w_smem, P.image + (size_t)unit0 * U * P.K * 2, (uint32_t)ncols * (uint32_t)P.K * 2u, bar(kWeights));
            }
            ok = mbar_wait(bar(kWeights), 0);
            int xb = 0, db = 0, it = 0;
            uint32_t xphase = 0, dphase = 1;
            for (int t = 0; ok && t < my_tiles; ++t) {
                if (!mbar_wait(bar(kXFull + xb), xphase)) { ok = false; break; }
                // The last tile is here: what follows sets itself up as blocks leave.  (In a load warp the line cost a register too many at
                // C = 256, 48 bytes of spills instead of 4.)
                if (P.early && t == my_tiles - 1) grid_launch_dependents();
                for (int ch = 0; ch < nchunks; ++ch, ++it) {
                    if (!mbar_wait(bar(kDFree + db), dphase)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t n = (uint32_t)(ncols - ch * kChunk < kChunk ? ncols - ch * kChunk : kChunk);
                    const uint32_t idesc = umma_idesc_bf16(128, n), d = tmem + kColD + (uint32_t)(db * kChunk), a = tmem + (uint32_t)(xb * 32 * NS);
                    const uint64_t b = umma_smem_desc(w_smem + (uint32_t)(ch * kChunk) * (uint32_t)P.K * 2u, 128, (uint32_t)P.K * 16u);
                    for (int kk = 0; kk < (P.K >> 4); ++kk) umma_bf16_ts(d, a + 8u * (uint32_t)kk, b + 16u * (uint32_t)kk, idesc, kk > 0 ? 1u : 0u);
                    umma_commit(bar(kDFull + db));
                    if (++db == kAccs) { db = 0; dphase ^= 1u; }
                }
                if (ok) umma_commit(bar(kXFree + xb));
                if (++xb == XB) { xb = 0; xphase ^= 1u; }
            }
            if (ok) ok = wait_last_phases(bar(kXFree), XB, my_tiles);       // no commit on its way when the block leaves
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else if (warp < kLoadWarps) {
        // ---- X: registers ahead, then tensor memory ---------------------------------------------------
        const uint32_t mine = tmem + ((uint32_t)(32 * (warp & 3) + 16 * (warp >> 2)) << 16);
        const int row_in_tile = 32 * (warp & 3) + 16 * (warp >> 2) + (lane >> 2), kunits = P.K / U;
        Pc x[TD][XU][2];
        auto load = [&](int t, Pc (&v)[XU][2]) {
            const long long row = ((long long)rank + (long long)t * nrank) * 128 + row_in_tile;
            const __nv_bfloat16* src = P.x + (size_t)row * P.K + (lane & 3) * (U / 4);
            const bool in[2] = {t < my_tiles && row < P.rows, t < my_tiles && row + 8 < P.rows};
#pragma unroll
            for (int u = 0; u < XU; ++u)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    v[u][r] = Pc();
                    if (u < kunits && in[r]) v[u][r] = *reinterpret_cast<const Pc*>(src + (size_t)(8 * r) * P.K + u * U);
                }
        };
#pragma unroll
        for (int j = 0; j < TD; ++j) load(j, x[j]);
        build();
        int xb = 0;
        uint32_t xphase = 1;
        for (int t0 = 0; ok && t0 < my_tiles; t0 += TD)
#pragma unroll
            for (int j = 0; j < TD; ++j) {
                if (!ok || t0 + j >= my_tiles) break;
                if (!warp_wait(bar(kXFree + xb), xphase)) { ok = false; break; }
                tc_fence_after_sync();
#pragma unroll
                for (int u = 0; u < XU; ++u)
                    if (u < kunits) store_x(mine + (uint32_t)(xb * 32 * NS + u * U / 2), x[j][u][0], x[j][u][1]);
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                mbar_arrive_lane0(bar(kXFull + xb), lane);
                if (++xb == XB) { xb = 0; xphase ^= 1u; }
                load(t0 + j + TD, x[j]);
            }
        if (!ok && lane == 0) atomicExch(P.status, 1);
    } else {
        // ---- Y ------------------------------------------------------------------------------------------
        const int w = warp - kLoadWarps, tig = lane & 3;
        const uint32_t mine = tmem + kColD + ((uint32_t)(32 * (w & 3) + 16 * (w >> 2)) << 16);
        const int row_in_tile = 32 * (w & 3) + 16 * (w >> 2) + (lane >> 2);
        build();
        const int mat0 = unit0 * U / P.ycols, col0 = unit0 * U - mat0 * P.ycols;
        int db = 0, it = 0;
        uint32_t dphase = 0;
        for (int t = 0; ok && t < my_tiles; ++t) {
            const long long row = ((long long)rank + (long long)t * nrank) * 128 + row_in_tile;
            const bool in[2] = {row < P.rows, row + 8 < P.rows};
            const size_t at = (size_t)row * P.ycols + tig * (U / 4);
            int mat = mat0, col = col0;
            for (int ch = 0; ch < nchunks; ++ch, ++it) {
                if (!warp_wait(bar(kDFull + db), dphase)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t d = mine + (uint32_t)(db * kChunk);
                uint32_t v[CU][U / 2];
#pragma unroll
                for (int u = 0; u < CU; ++u) {                   // past a narrow chunk's columns: not used
                    if constexpr (U == 32) tmem_ld_16x256b_x4_nowait(d + (uint32_t)(u * U), v[u]);
                    else tmem_ld_16x256b_x2_nowait(d + (uint32_t)(u * U), v[u]);
                }
                tmem_wait_ld();
#pragma unroll
                for (int u = 0; u < CU; ++u) tmem_pass(v[u]);
                tc_fence_before_sync();
                __syncwarp();
                mbar_arrive_lane0(bar(kDFree + db), lane);
#pragma unroll
                for (int u = 0; u < CU; ++u) {
                    if (ch * CU + u >= units) break;
                    __nv_bfloat16* dst = (mat == 0 ? P.y[0] : mat == 1 ? P.y[1] : P.y[2]) + at + col;
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        Pc o;
                        o.x = pack_bits(v[u][2 * r], v[u][2 * r + 1]);
                        o.y = pack_bits(v[u][4 + 2 * r], v[u][5 + 2 * r]);
                        if constexpr (U == 32) {
                            o.z = pack_bits(v[u][8 + 2 * r], v[u][9 + 2 * r]);
                            o.w = pack_bits(v[u][12 + 2 * r], v[u][13 + 2 * r]);
                        }
                        if (in[r]) *reinterpret_cast<Pc*>(dst + (size_t)(8 * r) * P.ycols) = o;
                    }
                    if ((col += U) == P.ycols) { col = 0; ++mat; }
                }
                if (++db == kAccs) { db = 0; dphase ^= 1u; }
            }
        }
        if (!ok && lane == 0) atomicExch(P.status, 1);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, 512);
    }
}

// Units of a group such that the bytes its busiest CTA moves, weights (w_bytes an element) and tiles, are fewest.
struct Split { int per_group, groups; long long ranks; };
Split split_columns(long long rows, int K, int units, int U, int w_bytes, int num_sms) {
    const long long ntiles = (rows + 127) / 128;
    Split s = {1, units, 1};
    long long best = -1;
    for (int per = units; per >= 1; --per) {
        const int groups = (units + per - 1) / per, cols = per * U;
        if ((uint32_t)cols * (uint32_t)K * 2u + kMisc > kMaxSmem || (groups > num_sms && per > 1)) continue;
        long long n = num_sms / groups > 0 ? num_sms / groups : 1;
        if (n > ntiles) n = ntiles;
        const long long cost = (long long)w_bytes * K * cols + (ntiles + n - 1) / n * 256 * (K + cols);
        if (best < 0 || cost < best) { best = cost; s = {per, groups, n}; }
    }
    return s;
}

int unit_of(int c_in, int c_out) { return c_in % 32 == 0 && c_out % 32 == 0 ? 32 : 16; }

using Kernel = void (*)(ProjParams);
template <int U, int NS>
Kernel configured_kernel() {                                     // null: the attribute could not be set
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    if (dev >= 64 || !configured[dev]) {
        if (cudaFuncSetAttribute(proj_kernel<U, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem) != cudaSuccess) return nullptr;
        if (dev < 64) configured[dev] = true;
    }
    return proj_kernel<U, NS>;
}
template <int U>
Kernel kernel_for(int K) {
    switch ((K + 63) / 64) {
        case 1: return configured_kernel<U, 1>();
        case 2: return configured_kernel<U, 2>();
        case 3: return configured_kernel<U, 3>();
        default: return configured_kernel<U, 4>();
    }
}

}  // namespace

bool proj_supports(int c_in, int c_out) {
    return c_in >= 16 && c_in <= 256 && c_in % 16 == 0 && c_out >= 16 && c_out <= 256 && c_out % 16 == 0;
}

// An image costs a launch, laying out in every CTA the time for 4 K cols bytes of fp32 weights (about 20 bytes a ns): up to 16 KB
// the latter is less.  A block call without and with images, us: 1 x 7 x 7 x 1 head (12 KB) 12.5 and 14.2; 64 x 40 x 40 x 1
// (12 KB) 28.4 and 28.5; 1 x 14 x 14 x 8 (32 KB) 16.5 and 14.7; 64 x 56 x 56 x 2 (48 KB) 60.5 and 59.0; 8 x 115 x 70 x 8 (384 KB)
// 128.8 and 92.2.
bool proj_wants_image(long long rows, int c_in, int c_out, int nmat, int num_sms) {
    const int U = unit_of(c_in, c_out);
    return 4LL * c_in * U * split_columns(rows, c_in, c_out * nmat / U, U, 4, num_sms).per_group > 16384;
}

size_t proj_image_bytes(int c_in, int c_out, int nmat) { return (size_t)c_in * c_out * nmat * 2; }

cudaError_t launch_proj_prep(const float* wa, int nmat_a, void* image_a, const float* wb, int nmat_b, void* image_b, int c_in, int c_out, cudaStream_t stream) {
    if (!proj_supports(c_in, c_out)) return cudaErrorInvalidValue;
    const int items = c_out * (nmat_a + nmat_b) * (c_in / 8);
    auto kernel = unit_of(c_in, c_out) == 32 ? proj_prep_kernel<32> : proj_prep_kernel<16>;
    return launch_chained(kernel, dim3((unsigned)((items + 255) / 256)), 256, 0, stream, wa, c_out * nmat_a, static_cast<unsigned char*>(image_a), wb,
                          c_out * nmat_b, static_cast<unsigned char*>(image_b), c_in, c_out);
}

cudaError_t launch_proj(const void* x, long long rows, int c_in, const float* w, const void* image, int c_out, int nmat,
                        void* const* y, bool early, int* d_status, int num_sms, cudaStream_t stream)
{
    if (!proj_supports(c_in, c_out) || nmat < 1 || nmat > 3 || rows < 1 || rows > 0x7fffff00LL) return cudaErrorInvalidValue;
    const int U = unit_of(c_in, c_out);
    ProjParams P;
    P.x = static_cast<const __nv_bfloat16*>(x); P.w = w; P.image = static_cast<const unsigned char*>(image);
    for (int i = 0; i < 3; ++i) P.y[i] = static_cast<__nv_bfloat16*>(i < nmat ? y[i] : nullptr);
    P.ycols = c_out; P.rows = (int)rows; P.K = c_in; P.units = c_out * nmat / U; P.status = d_status; P.early = early;
    const Split split = split_columns(rows, c_in, P.units, U, image ? 2 : 4, num_sms);
    P.per_group = split.per_group; P.groups = split.groups;
    const Kernel kernel = U == 32 ? kernel_for<32>(c_in) : kernel_for<16>(c_in);
    if (!kernel) return cudaErrorInvalidConfiguration;
    const uint32_t smem = (uint32_t)P.per_group * U * (uint32_t)c_in * 2u + kMisc;
    return launch_chained(kernel, dim3((unsigned)(split.ranks * split.groups)), kThreads, smem, stream, P);
}

}  // namespace slide_attn
