// UMMA_TS variant (bf16, head_dim 32, k = 3): BOTH contractions of the fused forward on the
// 5th-generation tensor core (tcgen05.mma), each with its A operand in tensor memory, so neither the
// q.k products nor the softmax weights pass through shared memory.
//
// Arithmetic (Eq. 2 with Eq. 12 inside; w = E + D, E the one-hot shift of Eq. 11):
//   product warps   P[p,(t,c)] = q[p,c] k[p+off(t),c]   packed bf16 multiply -> tcgen05.st (TMEM)
//   key MMA         L[p,n]     = sum_{t,c} P[p,(t,c)] Bk[(t,c),n]       tcgen05.mma, A from TMEM
//                   n = 0..8: deformed part D_k of slot n;  n = 9..17: plain q.k sum of tap n-9
//   softmax warps   logit[s] = (L[s] + L[9+s]) scale + bias[s];  e = exp2(logit - max) / sum_s exp2(logit - max)
//                   (tcgen05.ld.32x32b: one thread holds all logits of one pixel, no shuffles)
//                   A' row = e_hi | e_hi | e_lo | e8_hi e8_hi e8_lo 0..   -> tcgen05.st (TMEM)
//   value MMA       D[p,(t,c)] = sum_k A'[p,k] Bv[k,(t,c)]                     A from TMEM
//   value warps     out[p,c] = sum_t D[p,t,c] v[p+off(t),c]
//
// Persistent, one CTA per SM, CTA c -> head c mod heads.  A block is 128 pixels = four strips of 4 rows x 8 columns (team.cuh), which
// TMA brings with their halo (zero fill = the padding); blocks are dealt round-robin.  24 warps:
//   value warps    two sets of four; a set takes every other block, warp q of it strip q = quadrant q of tensor memory: lane (g, tig)
//                  works on column g and channels 8 tig .. of all four rows, so that each halo row is widened once for up to three of them
//   product warps  two sets likewise
//   softmax warps  four: thread = pixel
//   control warps  one thread each for the key MMAs, the value MMAs, the K and q strips, the head's weights and the V strips
// Registers move from the others to the value warps (setmaxnreg).  Waits of the compute warps have no vote and no way out (see
// wait_or_give_up).  Every wait is bounded; one that runs out sets the status word, and tensor memory is released on every path.
// Every CTA lays out its head's weights itself, in all warps but the control warps, while the first strips come: a prep launch in
// front cost 1 us at 64 x 56 x 56, 2 heads, and 1.7 us at 32 x 28 x 42, 6 heads.
//
// Tensor memory: three value chunks of 96 columns (dx), three P chunks of 48 (3 taps x 32 bf16), two logit tiles of 32, A' of 16.
//
// What bounds it: instruction issue and latency on the CUDA cores, and power in runs of seconds.  15.3 M warp instructions at 64 x 56 x 56,
// 2 heads, in 47 % of the slots (57 % while an SM has work); the value warps wait for 40 % of the time, the product warps for 50 %, so that no
// stage alone is the bound.  With value and product warps of two rows each on tiles of 4 rows x up to 64 columns it was 18.3 M (every
// halo row widened for two output rows instead of three, twice the hand-offs).  Calls, a few hundred / for seconds, when the power limit
// takes clocks down to 1.69 GHz here and 1.84 before: 64 x 56 x 56, 2 heads 32.3 / 34.0 -> 26.1 / 30.8 us, 32 x 28 x 42, 6 heads 23.5 / 23.4 ->
// 19.4 / 20.5, 2 x 56 x 56, 2 heads 7.9 -> 5.6.
// The code has to stay small: the instruction cache holds 32 KB, and a build of 112 KB (waits' spin loops and tile loops unrolled by
// the compiler) took 47 us.  Loops over tap columns not unrolled: 37 us.  fma.rn.f32x2 as two FMAs each: 3 % slower.  One set of
// product warps: 28.8; all of a chunk's accumulators read at once (160 registers): 29.6; two value chunks instead of three: the same.
#include "common.cuh"
#include "ptx.cuh"
#include "team.cuh"

namespace slide_attn {

namespace {

using team::Strips; using team::StripWalk; using team::kHaloPlane; using team::kSlot; using team::kLog2e;

constexpr int kHeadDim = 32;
constexpr int kVSets = 2, kPSets = 2;                    // of four value warps, of four product warps: they take the blocks in turn
constexpr int kPWarp0 = 4 * kVSets, kSWarp0 = kPWarp0 + 4 * kPSets, kCtlK = kSWarp0 + 4, kCtlV = kCtlK + 1, kCtlTK = kCtlK + 2, kCtlTV = kCtlK + 3;
constexpr int kThreads = (kCtlTV + 1) * 32;
constexpr int kLaunchRegs = 80, kValueRegs = 128, kProductRegs = 64, kSoftmaxRegs = 56, kControlRegs = 40;      // a thread: at the launch, then
static_assert(kVSets * kValueRegs + kPSets * kProductRegs + kSoftmaxRegs + kControlRegs <= kThreads / 128 * kLaunchRegs, "registers");
constexpr int kKSlots = 4, kVSlots = 6;
constexpr uint32_t kQStrip = 4 * 8 * 64;                // bytes of a strip of q
constexpr uint32_t kKSlot = kSlot + 4 * kQStrip;        // K with its halo, then q, of a block
constexpr int kBCols = 288;                             // value columns: (tap, channel)
constexpr int kBBytes = kBCols * 64;
constexpr int kBkBytes = 36 * 512;                      // key-side B: 288 K x 32 N bf16
constexpr int kImgBytes = kBBytes + kBkBytes;           // both B images of one head, as the prep kernel leaves them
constexpr int kWeightFloats = kHeadDim * 81;             // of a head, either side
constexpr uint32_t kTmemCols = 512;
// tensor-memory columns
constexpr uint32_t kColD = 0;                           // three value chunks of 96 columns
constexpr uint32_t kColP = 288;                         // three P chunks of 48 columns (3 taps x 32 bf16)
constexpr uint32_t kColL = 432, kOtherL = 96;           // two logit tiles of 32 columns, 432 and 432 ^ 96
constexpr uint32_t kColE = 496;                         // the A' tile of 16 columns (32 bf16)
constexpr uint32_t kIdesc96 = umma_idesc_bf16(128, 96);
constexpr uint32_t kIdesc32 = umma_idesc_bf16(128, 32);

struct UmmaParams {
    const float* wk;
    const float* wv;
    const unsigned char* bimg;       // per head: value-side B image (kBBytes) then key-side B image (kBkBytes); null: built here
    const float* bias;
    __nv_bfloat16* out;
    int* status;
    int H, W, heads;
    Strips strips;
    float scale_log2e;
};

// shared memory
constexpr uint32_t kVOff = kKSlots * kKSlot, kBOff = kVOff + kVSlots * (uint32_t)kSlot, kBkOff = kBOff + kBBytes, kBarOff = kBkOff + kBkBytes;

// barriers; those of a pair are told apart by bit 3 of their address
enum : int { kBarKFull = 0, kBarKEmpty = kBarKFull + kKSlots, kBarVFull = kBarKEmpty + kKSlots, kBarVEmpty = kBarVFull + kVSlots,
             kBarLFull = kBarVEmpty + kVSlots,           // [2] logits of a block complete
             kBarLFree = kBarLFull + 2,                  // [2] count 4: logits read
             kBarEReady = kBarLFree + 2, kBarEFree,      // count 4: A' rows stored; value MMAs of the block complete
             kBarDFree,                                  // [dx] count 4: value chunk read
             kBarDFull = kBarDFree + 3,                  // [set][dx] value chunk complete
             kBarPFree = kBarDFull + 3 * kVSets,         // [set][dx] key MMAs reading the chunk are complete
             kBarPReady = kBarPFree + 3 * kPSets,        // [dx] count 4: P chunk stored
             kBarWeights = kBarPReady + 3,               // count: the warps that build the images, or one for their copy
             kBarRaw,                                    // fp32 weights of the head
             kBars };
static_assert(kBarLFull % 2 == 0 && kKSlots % kPSets == 0 && kVSlots % kVSets == 0, "pairs of barriers; a slot has one set of readers");
constexpr uint32_t kTmemOff = kBarOff + 8 * kBars, kSmemBytes = kTmemOff + 16 + 128;
static_assert(kSmemBytes <= 227 * 1024, "shared memory");
// the fp32 weights wait in the last two slots of V, which V does not need before
constexpr int kRawSlots = 2;
constexpr uint32_t kRawOff = kVOff + (kVSlots - kRawSlots) * (uint32_t)kSlot;
static_assert(2 * kWeightFloats * 4 <= kRawSlots * kSlot, "fp32 weights");
constexpr int kBuilders = kCtlK;                        // all warps but the control warps

// Hand-offs of tensor memory between threads: the side that has read or written TMEM issues
// tcgen05.wait::ld / ::st (the accesses are then complete) and arrives on an mbarrier; the side that
// takes over waits on it and issues tcgen05.fence::after_thread_sync before its own tcgen05 work.

// ---------------------------------------------------------------------------------------------
// The two B images of a head, in the shared-memory layout the MMAs read (K-major core matrices of 8 rows x 16 bytes, no
// swizzle), from its fp32 weights [channel][slot][tap]; items of 16 bytes times 4 (value side) or 1 (key side).
//   value side  [288 columns][32 K] bf16: column n = (tap-column-major tap, channel); K rows
//               0..7 D_v[c][s][t], 8..15 and 16..23 the one-hot [s = t], 24 D_v[c][8][t], 25, 26 [t = 8]
//               (the A' row is e_hi | e_hi | e_lo | e8_hi e8_hi e8_lo)
//   key side    [288 K][32 N] bf16: K = 32 tap + kappa (kappa -> channel as tcgen05.st lays P out),
//               N 0..8 D_k[c][n][t], 9..17 the one-hot [n - 9 = t]
constexpr int kItems = kBCols + 36 * 32;
__device__ __forceinline__ void build_item(const float* wks, const float* wvs, unsigned char* sB, int item) {
    if (item < kBCols) {
        const int n = item;
        unsigned char* col = sB + (n >> 3) * 512 + (n & 7) * 16;
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = 0u;
        {
            const int ts = n >> 5, t = (ts % 3) * 3 + ts / 3;
            const int cn = n & 31, j = cn >> 3, wi = cn & 7;
            const float* wc = wvs + (8 * (wi >> 1) + 2 * j + (wi & 1)) * 81 + t;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int s0 = 2 * i, s1 = 2 * i + 1;
                w[i] = pack_bf16(wc[s0 * 9] - (s0 == t ? 1.f : 0.f), wc[s1 * 9] - (s1 == t ? 1.f : 0.f));
                const uint32_t oh = pack_bf16(s0 == t ? 1.f : 0.f, s1 == t ? 1.f : 0.f);
                w[4 + i] = oh; w[8 + i] = oh;
            }
            const float o8 = t == 8 ? 1.f : 0.f;
            w[12] = pack_bf16(wc[72] - o8, o8); w[13] = pack_bf16(o8, 0.f);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            *reinterpret_cast<uint4*>(col + c * 128) = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
    } else {
        const int it = item - kBCols;
        const int n = it & 31, kg = it >> 5;
        const int t = kg >> 2, kap0 = (kg & 3) * 8;
        float val[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int kap = kap0 + e;
            const int c = 8 * ((kap & 15) >> 2) + (kap & 3) + (kap >= 16 ? 4 : 0);
            float x = 0.f;
            if (n < 9) x = wks[c * 81 + n * 9 + t] - (n == t ? 1.f : 0.f);
            else if (n < 18) x = (n - 9 == t) ? 1.f : 0.f;
            val[e] = x;
        }
        *reinterpret_cast<uint4*>(sB + kBBytes + kg * 512 + (n >> 3) * 128 + (n & 7) * 16) =
            make_uint4(pack_bf16(val[0], val[1]), pack_bf16(val[2], val[3]), pack_bf16(val[4], val[5]), pack_bf16(val[6], val[7]));
    }
}

// The images of every head into the context workspace.  Only kernel timing launches this, which has to tell the attention from
// the layout of its weights; otherwise every CTA of the main kernel lays out its head's weights itself.
__global__ void __launch_bounds__(256)
umma_ts_prep_kernel(const float* __restrict__ wk, const float* __restrict__ wv, unsigned char* __restrict__ img)
{
    grid_dependency_wait();
    grid_launch_dependents();        // the main kernel may start its own prologue now
    const int h = blockIdx.x;
    for (int item = blockIdx.y * blockDim.x + threadIdx.x; item < kItems; item += gridDim.y * blockDim.x)
        build_item(wk + (size_t)h * kWeightFloats, wv + (size_t)h * kWeightFloats, img + (size_t)h * kImgBytes, item);
}

__global__ void __launch_bounds__(kThreads, 1)
umma_ts_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
               const __grid_constant__ CUtensorMap map_v, const UmmaParams P)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const uint32_t bar0 = smem_u32(smem + kBarOff);
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };

    // the warp index through a shuffle: the compiler then knows it is the same in every lane
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int h = blockIdx.x % P.heads, rank = blockIdx.x / P.heads, nrank = ((int)gridDim.x - h + P.heads - 1) / P.heads;
    const int blocks = (int)((P.strips.total + 3) >> 2);
    // blocks are dealt round-robin: neighbouring CTAs work on neighbouring blocks at the same time, which keeps the halos they
    // share in L2
    const int my_blocks = (blocks - rank + nrank - 1) / nrank;       // at least one: no head has more CTAs than blocks

    if (threadIdx.x < kBars) {                                     // a thread a barrier: one after the other they took 0.2 us
        const int i = threadIdx.x;
        auto in = [&](int first, int n) { return i >= first && i < first + n; };
        const bool warps = in(kBarKEmpty, kKSlots) || in(kBarVEmpty, kVSlots) || in(kBarLFree, 2) || i == kBarEReady || in(kBarDFree, 3) || in(kBarPReady, 3);
        mbar_init_only(bar(i), i == kBarWeights && !P.bimg ? (uint32_t)kBuilders : warps ? 4u : 1u);
        mbar_init_fence();
    }
    if (warp == kCtlK) tmem_alloc(smem_u32(smem + kTmemOff), kTmemCols);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *reinterpret_cast<const volatile uint32_t*>(smem + kTmemOff);
    bool ok = true;
    // the images of the weights, by the warps that wait for them to be used
    if (!P.bimg && warp < kBuilders) {
        wait_or_give_up(bar(kBarRaw), 0, ok);
        const float* raw = reinterpret_cast<const float*>(smem + kRawOff);
#pragma unroll 1
        for (int item = threadIdx.x; item < kItems; item += 32 * kBuilders) build_item(raw, raw + kWeightFloats, smem + kBOff, item);
        fence_proxy_async_smem();
        __syncwarp();
        mbar_arrive_lane0(bar(kBarWeights), lane);
    }

    if (warp < kPWarp0) {
        // =====================================================================================
        // value warps: set s takes blocks s, s + sets, ..; warp q of it strip q of the block
        // =====================================================================================
        reg_share<kValueRegs, kLaunchRegs>();
        const int q = warp & 3, set = warp >> 2, g = lane >> 2, tig = lane & 3;
        const uint32_t tq = tmem + kColD + ((uint32_t)(32 * q) << 16);
        const uint32_t full = bar(kBarDFull + 3 * set);
        const int C = P.heads * kHeadDim;
        const size_t row_pitch = (size_t)P.W * C;
        StripWalk walk(P.strips, 4LL * (rank + set * nrank) + q, 4LL * kVSets * nrank);
        const unsigned char* ring = smem + kVOff + (uint32_t)(q * kHaloPlane) + (uint32_t)g * 64u + (uint32_t)tig * 16u;
        const int last = (int)P.strips.total - q;
        const uint32_t zero = (uint32_t)(P.H >> 31);
        int slot = set;
        uint32_t phase = 0, parity = 0;                            // of the slot; of the chunks
#pragma unroll 1
        for (int blk = set; blk < my_blocks; blk += kVSets) {
            const unsigned char* src = ring + (uint32_t)slot * kSlot;
            wait_or_give_up(bar(kBarVFull + slot), phase, ok);
            float acc[4][8];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[i][c] = 0.f;
            uint4 vp[6];
#pragma unroll
            for (int r = 0; r < 6; ++r) vp[r] = lds128(src, (uint32_t)(r * 10) * 64u);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                wait_or_give_up(full + 8u * dx, parity, ok);
                tc_fence_after_sync();
                const uint32_t ta = tq + 96u * dx, tb = ta + (16u << 16);
                uint32_t d[48];
                tmem_ld3_16x256b_x4_nowait(ta, ta + 32, ta + 64, d);
                float vf[6][8];
                auto widen = [&](int r) {
                    const uint4 v = vp[r];
                    vf[r][0] = bf16_lo(v.x); vf[r][1] = bf16_hi(v.x); vf[r][2] = bf16_lo(v.y); vf[r][3] = bf16_hi(v.y);
                    vf[r][4] = bf16_lo(v.z); vf[r][5] = bf16_hi(v.z); vf[r][6] = bf16_lo(v.w); vf[r][7] = bf16_hi(v.w);
                };
                auto sum = [&](int m) {                            // pixel rows 2m, 2m + 1
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                ffma2(acc[2 * m + i][2 * j], acc[2 * m + i][2 * j + 1], __uint_as_float(d[16 * dy + 4 * j + 2 * i]),
                                      __uint_as_float(d[16 * dy + 4 * j + 2 * i + 1]), vf[2 * m + dy + i][2 * j], vf[2 * m + dy + i][2 * j + 1]);
                };
#pragma unroll
                for (int r = 0; r < 4; ++r) widen(r);
                tmem_wait_ld48(d);
                sum(0);
                tmem_ld3_16x256b_x4_nowait(tb, tb + 32, tb + 64, d);
                widen(4); widen(5);
                if (dx < 2)
#pragma unroll
                    for (int r = 0; r < 6; ++r) vp[r] = lds128(src, (uint32_t)(r * 10 + dx + 1) * 64u);
                tmem_wait_ld48(d);
                tc_fence_before_sync();
                mbar_arrive_lane0(bar(kBarDFree + dx), lane);
                sum(1);
            }
            mbar_arrive_lane0_after(bar(kBarVEmpty + slot), lane, acc[0][0], acc[3][0], zero);
            if ((slot += kVSets) >= kVSlots) { slot = set; phase ^= 1u; }
            parity ^= 1u;
            const int x = walk.x0() + g, y = walk.y0(), left = P.H - y;
            if (x < P.W && 4 * (rank + blk * nrank) < last) {
                __nv_bfloat16* op = P.out + (((size_t)walk.b * P.H + y) * P.W + x) * C + h * kHeadDim + tig * 8;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (i < left)
                        *reinterpret_cast<uint4*>(op + i * row_pitch) = make_uint4(pack_bf16(acc[i][0], acc[i][1]), pack_bf16(acc[i][2], acc[i][3]),
                                                                                   pack_bf16(acc[i][4], acc[i][5]), pack_bf16(acc[i][6], acc[i][7]));
            }
            walk.next();
        }
    } else if (warp < kSWarp0) {
        // =====================================================================================
        // product warps: as the value warps
        // =====================================================================================
        reg_share<kProductRegs, kLaunchRegs>();
        const int q = warp & 3, set = (warp - kPWarp0) >> 2, g = lane >> 2, tig = lane & 3;
        const uint32_t tq = tmem + kColP + ((uint32_t)(32 * q) << 16);
        const unsigned char* ring = smem + (uint32_t)g * 64u + (uint32_t)tig * 16u;
        // a chunk's buffer is free once the MMAs of the block before have read it, which the other set's barriers say
        const uint32_t free = bar(kBarPFree + 3 * ((set + kPSets - 1) % kPSets)), ready = bar(kBarPReady);
        int slot = set;
        uint32_t phase = 0, parity = set == 0 ? 1u : 0u;
#pragma unroll 1
        for (int blk = set; blk < my_blocks; blk += kPSets) {
            const unsigned char* sK = ring + (uint32_t)slot * kKSlot + (uint32_t)(q * kHaloPlane);
            const unsigned char* sQ = ring + (uint32_t)slot * kKSlot + (uint32_t)kSlot + (uint32_t)q * kQStrip;
            wait_or_give_up(bar(kBarKFull + slot), phase, ok);
            uint4 qf[4], kc[6];
#pragma unroll
            for (int i = 0; i < 4; ++i) qf[i] = lds128(sQ, (uint32_t)(i * 8) * 64u);
#pragma unroll
            for (int r = 0; r < 6; ++r) kc[r] = lds128(sK, (uint32_t)(r * 10) * 64u);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                wait_or_give_up(free + 8u * dx, parity, ok);
                tc_fence_after_sync();
#pragma unroll
                for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const uint4 q0 = qf[2 * m], q1 = qf[2 * m + 1], k0 = kc[2 * m + dy], k1 = kc[2 * m + dy + 1];
                        const uint32_t r[8] = {hmul2_bf16(q0.x, k0.x), hmul2_bf16(q0.y, k0.y), hmul2_bf16(q1.x, k1.x), hmul2_bf16(q1.y, k1.y),
                                               hmul2_bf16(q0.z, k0.z), hmul2_bf16(q0.w, k0.w), hmul2_bf16(q1.z, k1.z), hmul2_bf16(q1.w, k1.w)};
                        tmem_st_16x256b_x2(tq + ((uint32_t)(16 * m) << 16) + 48 * dx + 16 * dy, r);
                    }
                if (dx < 2)
#pragma unroll
                    for (int r = 0; r < 6; ++r) kc[r] = lds128(sK, (uint32_t)(r * 10 + dx + 1) * 64u);
                tmem_wait_st();
                tc_fence_before_sync();
                mbar_arrive_lane0(ready + 8u * dx, lane);
            }
            // the products that were made of what was read are in tensor memory
            mbar_arrive_lane0(bar(kBarKEmpty + slot), lane);
            if ((slot += kPSets) >= kKSlots) { slot = set; phase ^= 1u; }
            parity ^= 1u;
        }
    } else if (warp < kCtlK) {
        // =====================================================================================
        // softmax warps: thread = pixel = TMEM lane 32 q + lane, every block
        // =====================================================================================
        reg_share<kSoftmaxRegs, kLaunchRegs>();
        const uint32_t tq = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        grid_dependency_wait();
        float biasl[9];
#pragma unroll
        for (int s = 0; s < 9; ++s) biasl[s] = P.bias ? P.bias[h * 9 + s] * kLog2e : 0.f;
        uint32_t full = bar(kBarLFull), parity = 0, tl = tq + kColL;
#pragma unroll 1
        for (int blk = 0; blk < my_blocks; ++blk) {
            wait_or_give_up(full, parity, ok);
            tc_fence_after_sync();
            float Lg[18];
            tmem_ld_32x32b_18(tl, Lg);
            tc_fence_before_sync();
            mbar_arrive_lane0(full + 8u * (uint32_t)(kBarLFree - kBarLFull), lane);
            float l[9], m = -INFINITY;
#pragma unroll
            for (int s = 0; s < 9; ++s) { l[s] = (Lg[s] + Lg[9 + s]) * P.scale_log2e + biasl[s]; m = fmaxf(m, l[s]); }
            float e[9], sum = 0.f;
#pragma unroll
            for (int s = 0; s < 9; ++s) { e[s] = fast_exp2(l[s] - m); sum += e[s]; }
            const float inv = rcp_approx(sum);                     // the weights leave normalised: the value side only sums
            float hi[9], lo[9];
            uint32_t row[16];
#pragma unroll
            for (int s = 0; s < 9; ++s) {
                const float a = e[s] * inv;
                hi[s] = __bfloat162float(__float2bfloat16_rn(a));
                lo[s] = a - hi[s];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                row[i] = pack_bf16(hi[2 * i], hi[2 * i + 1]);
                row[4 + i] = row[i];
                row[8 + i] = pack_bf16(lo[2 * i], lo[2 * i + 1]);
            }
            row[12] = pack_bf16(hi[8], hi[8]);
            row[13] = pack_bf16(lo[8], 0.f);
            row[14] = row[15] = 0u;
            wait_or_give_up(bar(kBarEFree), ((uint32_t)blk & 1u) ^ 1u, ok);
            tc_fence_after_sync();
            tmem_st_32x32b_x16(tq + kColE, row);
            tmem_wait_st();
            tc_fence_before_sync();
            mbar_arrive_lane0(bar(kBarEReady), lane);
            full ^= 8u; tl ^= kOtherL;
            parity ^= (uint32_t)blk & 1u;
        }
    } else {
        reg_share<kControlRegs, kLaunchRegs>();
        // no copy or commit is on its way when the block leaves, whatever its readers have given up on; the barriers that are not
        // waited for here have readers that waited for their last phase
        auto drain = [&](int first, int slots, int uses) { ok = wait_last_phases(bar(first), slots, uses) && ok; };
        uint32_t leader;
        if (elect_one(leader)) {
            if (warp == kCtlK) {
                // ---- key MMAs: 18 per block (9 taps x two K = 16 halves) --------------------------------
                const uint64_t desc = umma_smem_desc(smem_u32(smem + kBkOff), 512, 128);
                const uint32_t b_lo = (uint32_t)desc, b_hi = (uint32_t)(desc >> 32);
                uint32_t full = bar(kBarLFull), parity = 0, dcol = tmem + kColL;
                int set = 0;
                ok = mbar_wait<true>(bar(kBarWeights), 0);
#pragma unroll 1
                for (int blk = 0; ok && blk < my_blocks; ++blk) {
                    if (!mbar_wait<true>(full + 8u * (uint32_t)(kBarLFree - kBarLFull), parity ^ 1u)) { ok = false; break; }
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        if (!mbar_wait<true>(bar(kBarPReady + dx), (uint32_t)blk & 1u)) { ok = false; break; }
                        tc_fence_after_sync();
#pragma unroll
                        for (int dy = 0; dy < 3; ++dy)
#pragma unroll
                            for (int kh = 0; kh < 2; ++kh)          // 16 bytes of descriptor address = 1 unit
                                umma_bf16_ts(dcol, tmem + kColP + 48 * dx + 16 * dy + 8 * kh, b_lo + (dx * 4 + dy * 12 + kh * 2) * 32, b_hi,
                                             kIdesc32, (dx != 0 || dy != 0 || kh != 0) ? 1u : 0u);
                        umma_commit(bar(kBarPFree + dx) + 24u * (uint32_t)set);
                        if (dx == 2) umma_commit(full);
                    }
                    if (kPSets == 2) set ^= 1;
                    full ^= 8u; dcol ^= kOtherL;
                    parity ^= (uint32_t)blk & 1u;
                }
                if (ok) drain(kBarPFree, 3 * kPSets, 3 * my_blocks);
            } else if (warp == kCtlV) {
                // ---- value MMAs -------------------------------------------------------------------------
                const uint64_t desc = umma_smem_desc(smem_u32(smem + kBOff), 128, 512);
                const uint32_t b_lo = (uint32_t)desc, b_hi = (uint32_t)(desc >> 32);
                uint32_t done = bar(kBarDFull);
                ok = mbar_wait<true>(bar(kBarWeights), 0);
#pragma unroll 1
                for (int blk = 0; ok && blk < my_blocks; ++blk) {
                    if (!mbar_wait<true>(bar(kBarEReady), (uint32_t)blk & 1u)) { ok = false; break; }
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        if (!mbar_wait<true>(bar(kBarDFree + dx), ((uint32_t)blk & 1u) ^ 1u)) { ok = false; break; }
                        tc_fence_after_sync();
                        const uint32_t dcol = tmem + kColD + 96u * dx;
                        umma_bf16_ts(dcol, tmem + kColE, b_lo + dx * 12 * 32, b_hi, kIdesc96, 0);
                        umma_bf16_ts(dcol, tmem + kColE + 8, b_lo + dx * 12 * 32 + 16, b_hi, kIdesc96, 1);
                        umma_commit(done + 8u * dx);
                        if (dx == 2) umma_commit(bar(kBarEFree));
                    }
                    if (kVSets == 2) done = done == bar(kBarDFull) ? done + 24u : bar(kBarDFull);
                }
                if (ok) drain(kBarEFree, 1, my_blocks);
            } else if (warp == kCtlTK) {
                // ---- K and q strips -----------------------------------------------------------------------
                grid_dependency_wait();
                StripWalk at(P.strips, 4LL * rank, 4LL * nrank);
                int slot = 0, blk = 0;
                uint32_t phase = 1;                                // a fresh barrier is free
#pragma unroll 1
                for (; blk < my_blocks; ++blk, at.next()) {
                    const uint32_t dst = smem_u32(smem) + (uint32_t)slot * kKSlot, full = bar(kBarKFull + slot);
                    if (!mbar_wait<true>(bar(kBarKEmpty + slot), phase)) { ok = false; break; }
                    mbar_expect_tx(full, kKSlot);
                    StripWalk s = at;                              // strips past the last one read as zero: their image does not exist
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        tma_load_4d(dst + (uint32_t)(i * kHaloPlane), &map_k, full, h * kHeadDim, s.x0() - 1, s.y0() - 1, s.b);
                        tma_load_4d(dst + (uint32_t)kSlot + (uint32_t)i * kQStrip, &map_q, full, h * kHeadDim, s.x0(), s.y0(), s.b);
                        if (++s.x == s.sx) { s.x = 0; if (++s.y == s.bands) { s.y = 0; ++s.b; } }
                    }
                    if (++slot == kKSlots) { slot = 0; phase ^= 1u; }
                }
                // What follows in the stream may be launched: as blocks leave, it takes their place and sets itself up.
                grid_launch_dependents();
                drain(kBarKFull, kKSlots, blk);
            } else {
                // ---- the head's weights, then V strips ------------------------------------------------------
                grid_dependency_wait();
                if (P.bimg) {
                    mbar_expect_tx(bar(kBarWeights), kImgBytes);
                    bulk_load_1d(smem_u32(smem + kBOff), P.bimg + (size_t)h * kImgBytes, kImgBytes, bar(kBarWeights));
                } else {
                    constexpr uint32_t bytes = kWeightFloats * 4;
                    mbar_expect_tx(bar(kBarRaw), 2 * bytes);
                    bulk_load_1d(smem_u32(smem + kRawOff), P.wk + (size_t)h * kWeightFloats, bytes, bar(kBarRaw));
                    bulk_load_1d(smem_u32(smem + kRawOff) + bytes, P.wv + (size_t)h * kWeightFloats, bytes, bar(kBarRaw));
                }
                StripWalk at(P.strips, 4LL * rank, 4LL * nrank);
                int slot = 0, blk = 0;
                uint32_t phase = 1;
#pragma unroll 1
                for (; blk < my_blocks; ++blk, at.next()) {
                    if (blk == kVSlots - kRawSlots && !mbar_wait<true>(bar(kBarWeights), 0)) { ok = false; break; }
                    if (!mbar_wait<true>(bar(kBarVEmpty + slot), phase)) { ok = false; break; }
                    team::load_strips(smem_u32(smem) + kVOff + (uint32_t)slot * kSlot, &map_v, bar(kBarVFull + slot), h * kHeadDim, at);
                    if (++slot == kVSlots) { slot = 0; phase ^= 1u; }
                }
                drain(kBarVFull, kVSlots, blk);
                if (blk <= kVSlots - kRawSlots) ok = mbar_wait<true>(bar(P.bimg ? kBarWeights : kBarRaw), 0) && ok;
            }
        }
        __syncwarp();
    }
    if (!ok) atomicExch(P.status, 1);
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kCtlK) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, kTmemCols);
    }
}

}  // namespace

bool umma_ts_supports(slide_attn_dtype dtype, int head_dim, int ksize) {
    return dtype == SLIDE_ATTN_BF16 && head_dim == kHeadDim && ksize == 3;
}

size_t umma_ts_workspace_bytes(int heads) { return (size_t)heads * kImgBytes; }

cudaError_t umma_ts_setup() {
    if (!tensor_map_available()) return cudaErrorNotSupported;
    return cudaFuncSetAttribute(umma_ts_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
}

cudaError_t launch_umma_ts_prep(const Problem& p, void* workspace, cudaStream_t stream) {
    return launch_chained(umma_ts_prep_kernel, dim3((unsigned)p.heads, 6), 256, 0, stream, p.wk, p.wv, static_cast<unsigned char*>(workspace));
}

// `workspace`: the images that launch_umma_ts_prep left there, or null.
cudaError_t launch_umma_ts(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream) {
    UmmaParams P;
    P.wk = p.wk; P.wv = p.wv; P.bimg = static_cast<const unsigned char*>(workspace); P.bias = p.bias;
    P.out = static_cast<__nv_bfloat16*>(p.out);
    P.status = d_status;
    P.H = p.H; P.W = p.W; P.heads = p.heads;
    P.strips.sx = (p.W + 7) / 8; P.strips.bands = (p.H + 3) / 4;
    P.strips.total = (long long)p.B * P.strips.bands * P.strips.sx;
    if (P.strips.total > 0x7fffffffLL - 4) return cudaErrorInvalidConfiguration;
    P.scale_log2e = kLog2e / sqrtf((float)kHeadDim);

    const int C = p.heads * kHeadDim;
    CUtensorMap map_q, map_k, map_v;
    if (!make_tile_map(&map_q, p.q, 2, p.B, p.H, p.W, C, kHeadDim, 8, 4) ||
        !make_tile_map(&map_k, p.k, 2, p.B, p.H, p.W, C, kHeadDim, 10, 6) ||
        !make_tile_map(&map_v, p.v, 2, p.B, p.H, p.W, C, kHeadDim, 10, 6))
        return cudaErrorInvalidValue;
    const long long blocks = (P.strips.total + 3) / 4;
    long long grid = num_sms > p.heads ? num_sms : p.heads;      // CTA c takes head c mod heads
    if (grid > blocks * p.heads) grid = blocks * p.heads;
    return launch_chained(umma_ts_kernel, dim3((unsigned)grid), kThreads, kSmemBytes, stream, map_q, map_k, map_v, P);
}

}  // namespace slide_attn
