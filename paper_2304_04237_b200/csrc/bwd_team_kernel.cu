// Backward pass for k = 3 (head_dim 32, fp32 or bf16 storage) on tcgen05 with fp32 arithmetic (split.cuh, team.cuh):
//
//   forward again   a = softmax_s( scale * sum_{t,c} q[c] k_t[c] wk[c,s,t] + bias[s] )
//   da[s]    = sum_{t,c} g[c] v_t[c] wv[c,s,t]                 (the logit contraction with g, v, wv)
//   dl[s]    = a[s] (da[s] - sum_s' a[s'] da[s'])              dbias[s] = sum over pixels of dl[s]
//   dq[c]    = scale * sum_t k_t[c] (sum_s dl[s] wk[c,s,t])    (the value expansion with dl, wk, k)
//   dk[p'][c] = scale * sum_t q[p' - off(t)][c] (sum_s dl[p' - off(t)][s] wk[c,s,t])
//   dv[p'][c] =         sum_t g[p' - off(t)][c] (sum_s  a[p' - off(t)][s] wv[c,s,t])
//
// bwd_point_kernel: two contractions, then one expansion, per query pixel; leaves dl and a as split rows.
// bwd_gather_kernel: dk and dv per key / value pixel, a gather over the nine query pixels whose window holds it.  The left
// operand of tap t is the split rows of the block's pixels moved by -off(t): every tap has rows of its own, copied from a halo
// in shared memory to tensor memory (out-of-map queries read as zero and contribute nothing), N = the channels of a plane.
// One launch computes both, or two launches one each where memory is short: the rows of dl then lie where dv will be (64 bytes a pixel and
// head, which is what dv takes in bf16) until the second launch writes it (64 x 56 x 56, 3 heads, bf16: 7 us more).
// Both persistent, one CTA per SM and one head per CTA, two teams; geometry and hand-offs as in umma_split_kernel.
//
// Bound by latency and instruction issue on the CUDA cores (products and their splits, sums, the point kernel's softmax, dL and row splits):
// at 64 x 56 x 56, 3 heads, bf16 the point kernel issues 64 M warp instructions in 48 % of the slots at 1.74 GHz, the gather kernel 46 M in 57 %;
// fp32 39 and 32 %.  64 x 56 x 56, 3 heads, bf16, in CUDA-core kernels before and here: point 333 and 131 us, gather 227 and 82; 2 x 128 x 128, 3
// heads, fp32: point 69 and 55, gather 54 and 24 us.
#include "bwd_common.cuh"
#include "team.cuh"

namespace slide_attn {

namespace {

using namespace team;

constexpr int kHeadDim = 32;
constexpr uint32_t kContract = contract_bytes(kHeadDim), kExpand = expand_bytes(kHeadDim);
// per head: contraction images of wk and wv, expansion images of wk and wv
constexpr uint32_t kImages = 2 * kContract + 2 * kExpand;
constexpr uint32_t kPointImages = 2 * kContract + kExpand, kGatherImages = 2 * kExpand, kGatherFrom = 2 * kContract;
constexpr uint32_t kMisc = 8u * (kTeams * kTeamBars + 1) + 16 + 2 * kK2 * 4 + 8;      // barriers, tensor-memory slot, bias, dbias

__host__ __device__ constexpr int ring_for(uint32_t images) {
    const int fit = (int)((227u * 1024u - images - kMisc - 128) / (kTeams * kSlot));
    return fit < kMaxRing ? fit : kMaxRing;
}
template <uint32_t Images> struct Plan {
    static constexpr int ring = ring_for(Images);
    static_assert(ring >= 4, "the ring does not fit");
    static constexpr uint32_t w_off = (uint32_t)(kTeams * ring * kSlot);
    static constexpr uint32_t bar_off = w_off + Images;
    static constexpr uint32_t total = bar_off + kMisc + 128;
};

struct TeamParams {
    const unsigned char* images;
    const void* q;
    const void* g;
    const float* bias;
    unsigned char* rows_dl;
    unsigned char* rows_a;
    void* dq;
    void* dk;
    void* dv;
    float* dbias;
    int* status;
    int H, W, heads;
    int first_side, sides;           // of bwd_gather_kernel: 0 dk, 1 dv
    Strips strips;
    float scale;
};

// Images of a head (blockIdx.x) and, spread over all blocks, zeros for what later kernels add to.  Comes right behind the forward of a
// training step, which lets it start early: spread over the SMs (launch_spread) a step of 8 x 56 x 56, 3 heads, bf16 takes 70.7 us,
// piled up 77.8; 3 x 54 x 54, 8 heads 75.0 and 84.0; 23 x 27 x 10, 3 heads, fp32 62.4 and 66.4.
// (One block an SM, for fp32, whose blocks take longer, two: 6 x 42 x 10, 4 heads, fp32 50.0 and 48.9, 4 x 28 x 28, 8 heads 63.2 and 62.8; 3 x 54 x 54,
// 8 heads, bf16 78.5 and 79.2.)
template <typename T>
__global__ void __launch_bounds__(256)
bwd_prep_kernel(const float* __restrict__ wk, const float* __restrict__ wv, unsigned char* __restrict__ images, float* dwk, float* dwv, float* dbias)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const size_t w = (size_t)blockIdx.x * kHeadDim * kK2 * kK2;
    unsigned char* img = images + (size_t)blockIdx.x * kImages;
    constexpr int contract_items = kHeadDim / 8 * kK2 * 48, expand_items = kHeadDim * kK2;
    const int step = gridDim.y * 256, at = blockIdx.y * 256 + threadIdx.x;
    float most[2] = {0.f, 0.f};
    const float* const both[2] = {wk + w, wv + w};
    if constexpr (sizeof(T) == 4) block_most<2>(both, kHeadDim * kK2 * kK2, most);
    for (int i = at; i < 2 * (contract_items + expand_items); i += step) {
        const int side = i >= contract_items + expand_items, j = side ? i - contract_items - expand_items : i;
        const float* src = both[side];
        if (j < contract_items) {
            float v[8];
            load_contract_item<T>(src, j, v);
            build_contract_item<T>(v, img + side * kContract, j, most[side]);
        } else {
            build_expand_item<T>(src, img + 2 * kContract + side * kExpand, j - contract_items);
        }
    }
    for (int i = at; i < kHeadDim * kK2 * kK2; i += step) { dwk[w + i] = 0.f; dwv[w + i] = 0.f; }
    if (dbias && at < kK2) dbias[blockIdx.x * kK2 + at] = 0.f;
}

// Eight (bf16) or four (fp32) channels of a pixel to memory.
__device__ __forceinline__ void store_piece(__nv_bfloat16* p, const float (&f)[8], float s) {
    *reinterpret_cast<uint4*>(p) = make_uint4(pack_bf16(f[0] * s, f[1] * s), pack_bf16(f[2] * s, f[3] * s), pack_bf16(f[4] * s, f[5] * s),
                                              pack_bf16(f[6] * s, f[7] * s));
}
__device__ __forceinline__ void store_piece(float* p, const float (&f)[4], float s) {
    *reinterpret_cast<float4*>(p) = make_float4(f[0] * s, f[1] * s, f[2] * s, f[3] * s);
}

// What both kernels share: the CTA's set-up and its geometry.
struct Seat {
    int warp, lane, h, team_id, first, step, my_blocks;
    uint32_t bars, bar_weights, tmem;
    unsigned char* ring;
    __device__ __forceinline__ uint32_t bar(int i) const { return bars + 8u * (uint32_t)(team_id * kTeamBars + i); }
    __device__ __forceinline__ long long strip0(int bi) const { return 4LL * (first + (long long)bi * step); }
};
template <uint32_t Images>
__device__ __forceinline__ Seat take_seat(unsigned char* smem, const TeamParams& P) {
    using L = Plan<Images>;
    Seat s;
    s.warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); s.lane = threadIdx.x & 31;
    s.h = blockIdx.x % P.heads;
    const int rank = blockIdx.x / P.heads, nrank = (int)gridDim.x / P.heads;
    s.team_id = s.warp < kComputeWarps ? s.warp / kTeamWarps : (s.warp - kComputeWarps) % kTeams;
    const int blocks = (int)((P.strips.total + 3) >> 2);
    s.first = s.team_id * nrank + rank; s.step = kTeams * nrank;
    s.my_blocks = s.first < blocks ? (blocks - s.first + s.step - 1) / s.step : 0;
    s.bars = smem_u32(smem + L::bar_off);
    s.bar_weights = s.bars + 8u * (kTeams * kTeamBars);
    s.ring = smem + (uint32_t)(s.team_id * L::ring * kSlot);
    unsigned char* tmem_slot = smem + L::bar_off + 8u * (kTeams * kTeamBars + 1);
    if (threadIdx.x == 0) {
        for (int i = 0; i < kTeams; ++i) init_team_bars(s.bars + 8u * (uint32_t)(i * kTeamBars));
        mbar_init_only(s.bar_weights, 1);
        mbar_init_fence();
    }
    if (s.warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    s.tmem = *reinterpret_cast<const volatile uint32_t*>(tmem_slot) + kCols * (uint32_t)s.team_id;
    return s;
}
template <uint32_t Images>
__device__ __forceinline__ void leave_seat(unsigned char* smem, const Seat& s) {
    tc_fence_before_sync();
    __syncthreads();
    if (s.warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(*reinterpret_cast<const volatile uint32_t*>(smem + Plan<Images>::bar_off + 8u * (kTeams * kTeamBars + 1)), 512);
    }
}
// The pixels of a compute lane: two rows of column g of a strip.
struct Place { size_t pix; bool in[2]; };
struct Lane {
    StripWalk walk;
    int wq, half, g, tig;
    __device__ __forceinline__ Lane(const Seat& s, const TeamParams& P)
        : walk(P.strips, s.strip0(0) + (s.warp & 3), 4LL * s.step), wq(s.warp & 3), half(s.warp % kTeamWarps >> 2), g(s.lane >> 2), tig(s.lane & 3) {}
    // pixel (row, column) of the walk's strip, which is strip `i`, and the one below it; nothing is inside past the last strip
    __device__ __forceinline__ Place place(const TeamParams& P, long long i, int row, int col) const {
        Place p;
        const int y = walk.y0() + row, x = walk.x0() + col;
        const bool in = i < P.strips.total && x < P.W;
        p.in[0] = in && y < P.H; p.in[1] = in && y + 1 < P.H;
        p.pix = ((size_t)walk.b * P.H + y) * P.W + x;
        return p;
    }
};

template <typename T>
__global__ void __launch_bounds__(kThreads, 1)
bwd_point_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const TeamParams P)
{
    using L = Plan<kPointImages>;
    constexpr int CH = Cut<T>::channels, NPL = kHeadDim / CH, PL = Cut<T>::per_lane, DB = Cut<T>::d_buffers, R = L::ring, CHUNKS = 3 * NPL;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    float* s_bias = reinterpret_cast<float*>(smem + L::bar_off + 8u * (kTeams * kTeamBars + 1) + 16);
    float* s_dbias = s_bias + kK2;
    if (threadIdx.x < kK2) {
        s_bias[threadIdx.x] = P.bias ? P.bias[(blockIdx.x % P.heads) * kK2 + threadIdx.x] * kLog2e : 0.f;
        s_dbias[threadIdx.x] = 0.f;
    }
    const Seat seat = take_seat<kPointImages>(smem, P);
    auto bar = [&](int i) { return seat.bar(i); };
    const int warp = seat.warp, lane = seat.lane, h = seat.h, my_blocks = seat.my_blocks;
    const uint32_t tmem = seat.tmem;
    bool ok = true;

    if (warp >= kTmaWarp) {
        // ---- TMA thread of a team: K, V and K again ------------------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            int slot = 0;
            uint32_t phase = 1;
            StripWalk at(P.strips, seat.strip0(0), 4LL * seat.step);
            for (int bi = 0; ok && bi < my_blocks; ++bi, at.next()) {
                for (int v = 0; v < 3 * NPL; ++v) {
                    if (!mbar_wait(bar(kEmpty + slot), phase)) { ok = false; break; }
                    load_strips(smem_u32(seat.ring) + (uint32_t)(slot * kSlot), v / NPL == 1 ? &map_v : &map_k, bar(kFull + slot), h * kHeadDim + (v % NPL) * CH, at);
                    if (++slot == R) { slot = 0; phase ^= 1u; }
                }
            }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else if (warp >= kMmaWarp) {
        // ---- MMA thread of a team ------------------------------------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            const uint32_t w = smem_u32(smem + L::w_off);
            if (warp == kMmaWarp) {
                grid_dependency_wait();
                mbar_expect_tx(seat.bar_weights, kPointImages);
                bulk_load_1d(w, P.images + (size_t)h * kImages, kPointImages, seat.bar_weights);
            }
            if (my_blocks > 0) ok = mbar_wait(seat.bar_weights, 0);
            const uint32_t dsrc = w + 2 * kContract;
            int pn = 0, dn = 0;
            for (int bi = 0; ok && bi < my_blocks; ++bi) {
                for (int side = 0; ok && side < 2; ++side) {
                    const uint64_t desc = contract_desc(w + side * kContract);
                    for (int i = 0; i < CHUNKS; ++i, ++pn) {             // plane, tap column
                        const int pb = pn & 1, plane = i / 3, dx = i % 3;
                        if (!mbar_wait(bar(kPFull + pb), (uint32_t)(pn >> 1) & 1u)) { ok = false; break; }
                        if (side == 1 && i == 0 && !mbar_wait(bar(kLFree), (uint32_t)bi & 1u)) { ok = false; break; }
                        tc_fence_after_sync();
                        const uint32_t p_col = tmem + kColP + (uint32_t)(pb * 3 * Cut<T>::tap_cols);
#pragma unroll
                        for (int dy = 0; dy < 3; ++dy)
                            issue_contract<T>(tmem, p_col + dy * Cut<T>::tap_cols, desc + contract_step<T>(plane, dy * 3 + dx), plane, dx, dy);
                        umma_commit(bar(kPFree + pb));
                    }
                    if (ok) umma_commit(bar(kLFull));
                }
                if (!ok || !mbar_wait(bar(kAFull), (uint32_t)bi & 1u)) { ok = false; break; }
                for (int i = 0; i < CHUNKS; ++i, ++dn) {
                    const int db = dn % DB;
                    if (!mbar_wait(bar(kDFree + db), ((uint32_t)(dn / DB) & 1u) ^ 1u)) { ok = false; break; }
                    tc_fence_after_sync();
                    issue_expand<3 * CH>(tmem + kColD + (uint32_t)(db * 3 * CH), tmem + kColA, dsrc + (uint32_t)(i * 3 * CH * 128));
                    umma_commit(bar(kDFull + db));
                }
            }
            if (ok) ok = wait_last_phases(bar(kPFree), 2, pn);      // no commit on its way when the block leaves
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else {
        Lane me(seat, P);
        const int wq = me.wq, half = me.half, g = me.g, tig = me.tig;
        const uint32_t quad = tmem + ((uint32_t)(32 * wq) << 16), mine = quad + ((uint32_t)(16 * half) << 16);
        const int C = P.heads * kHeadDim, piece = h * kHeadDim + tig * PL;
        const size_t row_pitch = (size_t)P.W * C;
        float dbias[kK2];
#pragma unroll
        for (int s = 0; s < kK2; ++s) dbias[s] = 0.f;
        int slot = 0, pn = 0, dn = 0;
        uint32_t phase = 0;
        const uint32_t zero = (uint32_t)(P.H >> 31);
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
        auto load_x = [&](const Place& p, int side, int plane, uint4 (&x)[2]) {
            const T* src = static_cast<const T*>(side ? P.g : P.q) + p.pix * C + piece + plane * CH;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                x[r] = make_uint4(0u, 0u, 0u, 0u);
                if (p.in[r]) x[r] = __ldg(reinterpret_cast<const uint4*>(src + r * row_pitch));
            }
        };
        Place st = me.place(P, seat.strip0(0) + wq, 2 * half, g);
        uint4 xn[2];
        if (my_blocks > 0) load_x(st, 0, 0, xn);
        for (int bi = 0; ok && bi < my_blocks; ++bi) {
            const bool turn = half == (bi & 1);                      // the warps that do the softmax of this block
            float a[kK2];
            // ---- products of both sides ----------------------------------------------------------------
            for (int v = 0; v < 2 * NPL; ++v) {
                Factor<T> x;
                x.set(xn);
                if (v + 1 < 2 * NPL) load_x(st, (v + 1) / NPL, (v + 1) % NPL, xn);
                if (!warp_wait(bar(kFull + slot), phase)) { ok = false; break; }
                const unsigned char* plane = seat.ring + (uint32_t)(slot * kSlot + wq * kHaloPlane);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx, ++pn) {
                    const int pb = pn & 1;
                    uint4 y[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) y[r] = halo_piece<T>(plane, 2 * half + r, g + dx, tig);
                    if (dx == 0) x.meet(plane, 2 * half, g, tig, y);
                    if (!warp_wait(bar(kPFree + pb), ((uint32_t)(pn >> 1) & 1u) ^ 1u)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t t = mine + kColP + (uint32_t)(pb * 3 * Cut<T>::tap_cols);
                    store_column<T>(x, t, y);
                    tmem_wait_st();
                    tc_fence_before_sync();
                    __syncwarp();
                    mbar_arrive_lane0(bar(kPFull + pb), lane);
                    // the logits: complete while the first chunk of the other side was made
                    if (dx == 0 && v == NPL && turn) {
                        if (!warp_wait(bar(kLFull), 0)) { ok = false; break; }
                        tc_fence_after_sync();
                        load_contraction<T>(quad, a);
                        tc_fence_before_sync();
                        __syncwarp();
                        mbar_arrive_lane0(bar(kLFree), lane);
                    }
                }
                if (!ok) break;
                release();
            }
            if (!ok) break;
            const Place cur = st;

            // ---- a and dl: thread = pixel of the quadrant ------------------------------------------------
            if (turn) {
                const float iz = 1.f / softmax_terms(a, P.scale * kLog2e, s_bias);
#pragma unroll
                for (int s = 0; s < kK2; ++s) a[s] *= iz;
                // lane = 8 row + column of the strip
                const Place px = me.place(P, seat.strip0(bi) + wq, lane >> 3, lane & 7);
                // Lanes 2i and 2i + 1 write both pieces of a 32-byte sector together: piece c of the even lane's pixel and its
                // neighbour c + 1, then of the odd one's (16 bytes of each sector at a time took 20 of the kernel's 132 us).
                const size_t at = (px.pix * P.heads + h) * 64, pitch = (size_t)P.heads * 64;
                const bool odd = lane & 1, other = __shfl_xor_sync(0xffffffffu, (int)px.in[0], 1) != 0;
                const bool in_even = odd ? other : px.in[0], in_odd = odd ? px.in[0] : other;
                const size_t at_even = odd ? at - pitch : at;
                const uint32_t swz = (uint32_t)(lane >> 1) & 3u;                 // x0 is a multiple of 8
                auto write = [&](unsigned char* rows, const uint32_t (&w)[16]) {
#pragma unroll
                    for (uint32_t m = 0; m < 2; ++m) {                           // pieces 2m, 2m + 1
                        uint32_t e[4], o[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint32_t lo = w[8 * m + i], hi = w[8 * m + 4 + i], got = __shfl_xor_sync(0xffffffffu, odd ? lo : hi, 1);
                            e[i] = odd ? got : lo;                               // of the even pixel: this lane's piece 2m + odd
                            o[i] = odd ? hi : got;                               // of the odd pixel
                        }
                        const uint32_t c = ((2 * m + (odd ? 1u : 0u)) ^ swz) << 4;
                        if (in_even) *reinterpret_cast<uint4*>(rows + at_even + c) = make_uint4(e[0], e[1], e[2], e[3]);
                        if (in_odd) *reinterpret_cast<uint4*>(rows + at_even + pitch + c) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                };
                uint32_t row[16];
                split_row(a, row);
                write(P.rows_a, row);                                // while the other side's last MMAs run
                if (!warp_wait(bar(kLFull), 1)) { ok = false; break; }
                tc_fence_after_sync();
                float dl[kK2], mean = 0.f;
                load_contraction<T>(quad, dl);                       // da
#pragma unroll
                for (int s = 0; s < kK2; ++s) mean = fmaf(a[s], dl[s], mean);
#pragma unroll
                for (int s = 0; s < kK2; ++s) dl[s] = a[s] * (dl[s] - mean);
                split_row(dl, row);
                tmem_st_32x32b_x16(quad + kColA, row);
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                mbar_arrive_lane0(bar(kAFull), lane);
                if (px.in[0]) {
#pragma unroll
                    for (int s = 0; s < kK2; ++s) dbias[s] += dl[s];
                }
                write(P.rows_dl, row);
            }

            if (bi + 1 < my_blocks) { me.walk.next(); st = me.place(P, seat.strip0(bi + 1) + wq, 2 * half, g); load_x(st, 0, 0, xn); }

            // ---- dq ----------------------------------------------------------------------------------
            for (int pl = 0; pl < NPL; ++pl) {
                float acc[2][PL];
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int c = 0; c < PL; ++c) acc[r][c] = 0.f;
                if (!warp_wait(bar(kFull + slot), phase)) { ok = false; break; }
                const unsigned char* plane = seat.ring + (uint32_t)(slot * kSlot + wq * kHaloPlane);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx, ++dn) {
                    const int db = dn % DB;
                    if (!warp_wait(bar(kDFull + db), (uint32_t)(dn / DB) & 1u)) { ok = false; break; }
                    tc_fence_after_sync();
                    sum_chunk(T(), mine + kColD + (uint32_t)(db * 3 * CH), plane, 2 * half, g + dx, tig, acc);
                    tc_fence_before_sync();
                    __syncwarp();
                    mbar_arrive_lane0(bar(kDFree + db), lane);
                }
                if (!ok) break;
                release_after(acc[0][0], acc[1][0]);
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    if (cur.in[r]) store_piece(static_cast<T*>(P.dq) + cur.pix * C + piece + pl * CH + r * row_pitch, acc[r], P.scale);
            }
        }
        if (!ok && lane == 0) atomicExch(P.status, 1);
        if (P.dbias) {
#pragma unroll
            for (int s = 0; s < kK2; ++s) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) dbias[s] += __shfl_xor_sync(0xffffffffu, dbias[s], o);
                if (lane == 0) atomicAdd(&s_dbias[s], dbias[s]);
            }
        }
    }
    leave_seat<kPointImages>(smem, seat);
    if (P.dbias && threadIdx.x < kK2) atomicAdd(&P.dbias[h * kK2 + threadIdx.x], s_dbias[threadIdx.x]);
}

// Tensor memory of a team here: D chunks in 0 - 191, the left operands of a tap column's three taps in 192 - 239.
template <typename T>
__global__ void __launch_bounds__(kThreads, 1)
bwd_gather_kernel(const __grid_constant__ CUtensorMap map_dl, const __grid_constant__ CUtensorMap map_a,
                  const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_g, const TeamParams P)
{
    using L = Plan<kGatherImages>;
    constexpr int CH = Cut<T>::channels, NPL = kHeadDim / CH, PL = Cut<T>::per_lane, DB = Cut<T>::d_buffers, R = L::ring;
    constexpr uint32_t kColRows = 192;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const Seat seat = take_seat<kGatherImages>(smem, P);
    auto bar = [&](int i) { return seat.bar(i); };
    const int warp = seat.warp, lane = seat.lane, h = seat.h, my_blocks = seat.my_blocks;
    const uint32_t tmem = seat.tmem;
    bool ok = true;

    if (warp >= kTmaWarp) {
        // ---- TMA thread of a team: per side the rows, then the planes ---------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            grid_dependency_wait();                                  // the rows come from the kernel before
            int slot = 0;
            uint32_t phase = 1;
            StripWalk at(P.strips, seat.strip0(0), 4LL * seat.step);
            for (int bi = 0; ok && bi < my_blocks; ++bi, at.next()) {
                for (int v = 0; v < P.sides * (NPL + 1); ++v) {
                    const int side = P.first_side + v / (NPL + 1), pl = v % (NPL + 1) - 1;
                    if (!mbar_wait(bar(kEmpty + slot), phase)) { ok = false; break; }
                    load_strips(smem_u32(seat.ring) + (uint32_t)(slot * kSlot), pl < 0 ? (side ? &map_a : &map_dl) : (side ? &map_g : &map_q), bar(kFull + slot),
                                h * kHeadDim + (pl < 0 ? 0 : pl * CH), at);
                    if (++slot == R) { slot = 0; phase ^= 1u; }
                }
            }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else if (warp >= kMmaWarp) {
        // ---- MMA thread of a team ------------------------------------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            const uint32_t w = smem_u32(smem + L::w_off);
            if (warp == kMmaWarp) {
                grid_dependency_wait();
                mbar_expect_tx(seat.bar_weights, kGatherImages);
                bulk_load_1d(w, P.images + (size_t)h * kImages + kGatherFrom, kGatherImages, seat.bar_weights);
            }
            if (my_blocks > 0) ok = mbar_wait(seat.bar_weights, 0);
            int dn = 0;
            for (int s = 0; ok && s < my_blocks * P.sides * 3; ++s) { // side, tap column
                const int side = P.first_side + (s / 3 & (P.sides - 1)), dx = s % 3;
                if (!mbar_wait(bar(kAFull), (uint32_t)s & 1u)) { ok = false; break; }
                for (int pl = 0; pl < NPL; ++pl, ++dn) {
                    const int db = dn % DB;
                    if (!mbar_wait(bar(kDFree + db), ((uint32_t)(dn / DB) & 1u) ^ 1u)) { ok = false; break; }
                    tc_fence_after_sync();
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy)
                        issue_expand<CH>(tmem + kColD + (uint32_t)(db * 3 * CH + dy * CH), tmem + kColRows + 16 * dy,
                                          w + side * kExpand + (uint32_t)(((pl * 3 + dx) * 3 + dy) * CH * 128));
                    umma_commit(bar(kDFull + db));
                }
            }
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else {
        Lane me(seat, P);
        const int wq = me.wq, half = me.half, g = me.g, tig = me.tig;
        const uint32_t quad = tmem + ((uint32_t)(32 * wq) << 16), mine = quad + ((uint32_t)(16 * half) << 16);
        const int C = P.heads * kHeadDim, piece = h * kHeadDim + tig * PL;
        const size_t row_pitch = (size_t)P.W * C;
        // visit v of the stream of planes (NPL + 1 per side): slot v % R, phase v / R
        int rows_slot = 0;
        uint32_t rows_phase = 0;
        auto ahead = [](int& slot, uint32_t& phase, int by) { slot += by; if (slot >= R) { slot -= R; phase ^= 1u; } };
        const uint32_t rows_at = (uint32_t)(wq * kHaloPlane) + (uint32_t)(((lane >> 3) + 2) * 10 + (lane & 7) + 2) * 64u;
        // the left operands of a step (tap column dx; `turn`: this warp's): pixel (row, column) of the strip reads halo pixel
        // (row + 2 - dy, column + 2 - dx)
        auto store_rows = [&](int dx, bool turn) -> bool {
            if (dx == 0 && !warp_wait(bar(kFull + rows_slot), rows_phase)) return false;
            if (turn) {
                const uint32_t swz = (uint32_t)(((lane & 7) + 1 - dx) >> 1) & 3u;
                const unsigned char* src = seat.ring + (uint32_t)(rows_slot * kSlot) + rows_at - dx * 64;
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    uint32_t row[16];
#pragma unroll
                    for (uint32_t c = 0; c < 4; ++c) {
                        const uint4 v = *reinterpret_cast<const uint4*>(src - dy * 640 + ((c ^ swz) << 4));
                        row[4 * c] = v.x; row[4 * c + 1] = v.y; row[4 * c + 2] = v.z; row[4 * c + 3] = v.w;
                    }
                    tmem_st_32x32b_x16(quad + kColRows + 16 * dy, row);
                }
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                mbar_arrive_lane0(bar(kAFull), lane);
            }
            if (dx == 2) {
                __syncwarp();
                mbar_arrive_lane0(bar(kEmpty + rows_slot), lane);
                ahead(rows_slot, rows_phase, NPL + 1);
            }
            return true;
        };
        int slot = 1, dn = 0;                                        // of the side's first plane
        uint32_t phase = 0;
        if (my_blocks > 0) ok = store_rows(0, half == 0);
        const int steps = P.sides * my_blocks;
        for (int bs = 0; ok && bs < steps; ++bs) {                   // block, side
            const int side = P.first_side + (bs & (P.sides - 1));
            const bool even = half == (bs & 1);                      // step 3 bs + dx is this warp's if even == (dx != 1)
            float acc[NPL][2][PL];
#pragma unroll
            for (int pl = 0; pl < NPL; ++pl)
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int c = 0; c < PL; ++c) acc[pl][r][c] = 0.f;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                int ps = slot;
                uint32_t pp = phase;
#pragma unroll
                for (int pl = 0; pl < NPL; ++pl, ++dn) {
                    const int db = dn % DB;
                    if (dx == 0 && !warp_wait(bar(kFull + ps), pp)) { ok = false; break; }
                    if (!warp_wait(bar(kDFull + db), (uint32_t)(dn / DB) & 1u)) { ok = false; break; }
                    tc_fence_after_sync();
                    // the last MMAs of this step are complete: its operands make room for the next ones
                    if (pl == NPL - 1) {
                        if (dx < 2) { if (!store_rows(dx + 1, dx == 0 ? !even : even)) { ok = false; break; } }
                        else if (bs + 1 < steps) { if (!store_rows(0, !even)) { ok = false; break; } }
                    }
                    sum_chunk<true>(T(), mine + kColD + (uint32_t)(db * 3 * CH), seat.ring + (uint32_t)(ps * kSlot + wq * kHaloPlane), 2 * half, g + 2 - dx, tig, acc[pl]);
                    tc_fence_before_sync();
                    __syncwarp();
                    mbar_arrive_lane0(bar(kDFree + db), lane);
                    if (dx == 2) mbar_arrive_lane0_after(bar(kEmpty + ps), lane, acc[pl][0][0], acc[pl][1][0], (uint32_t)(P.H >> 31));
                    ahead(ps, pp, 1);
                }
                if (!ok) break;
            }
            if (!ok) break;
            ahead(slot, phase, NPL + 1);
            const Place p = me.place(P, seat.strip0(P.sides == 2 ? bs >> 1 : bs) + wq, 2 * half, g);
            T* out = static_cast<T*>(side ? P.dv : P.dk) + p.pix * C + piece;
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (p.in[r])
#pragma unroll
                    for (int pl = 0; pl < NPL; ++pl) store_piece(out + r * row_pitch + pl * CH, acc[pl][r], side ? 1.f : P.scale);
            if (side || P.sides == 1) me.walk.next();
        }
        if (!ok && lane == 0) atomicExch(P.status, 1);
    }
    leave_seat<kGatherImages>(smem, seat);
}

template <typename T>
cudaError_t launch_t(BwdPass what, const Problem& p, const BackwardArgs& ga, const BwdScratch& ws, int* d_status, int num_sms, cudaStream_t stream) {
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(bwd_point_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Plan<kPointImages>::total);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(bwd_gather_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Plan<kGatherImages>::total);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured[dev] = true;
    }
    TeamParams P;
    P.images = ws.images; P.q = p.q; P.g = ga.dout; P.bias = p.bias; P.rows_dl = ws.rows_dl; P.rows_a = ws.rows_a;
    P.dq = ga.dq; P.dk = ga.dk; P.dv = ga.dv; P.dbias = ga.dbias; P.status = d_status;
    P.H = p.H; P.W = p.W; P.heads = p.heads;
    P.strips.sx = (p.W + 7) / 8; P.strips.bands = (p.H + 3) / 4;
    P.strips.total = (long long)p.B * P.strips.bands * P.strips.sx;
    if (P.strips.total > 0x7fffffffLL - 4) return cudaErrorInvalidConfiguration;
    P.scale = 1.f / sqrtf((float)kHeadDim);
    P.first_side = 0; P.sides = 2;
    const int C = p.heads * kHeadDim, es = (int)sizeof(T), ch = Cut<T>::channels;
    const long long blocks = (P.strips.total + 3) / 4;
    long long per_head = num_sms / p.heads;
    if (per_head > blocks) per_head = blocks;
    if (per_head < 1) per_head = 1;
    const dim3 grid((unsigned)(per_head * p.heads));
    if (what == BwdPass::point) {
        CUtensorMap mk, mv;
        if (!make_tile_map(&mk, p.k, es, p.B, p.H, p.W, C, ch, 10, 6) || !make_tile_map(&mv, p.v, es, p.B, p.H, p.W, C, ch, 10, 6)) return cudaErrorInvalidValue;
        e = launch_spread<bwd_prep_kernel<T>, sizeof(T) == 4 ? 2 : 1>(dim3((unsigned)p.heads, 9), 256, stream, p.wk, p.wv, ws.images, ga.dwk, ga.dwv, ga.dbias);
        if (e != cudaSuccess) return e;
        return launch_chained(bwd_point_kernel<T>, grid, kThreads, Plan<kPointImages>::total, stream, mk, mv, P);
    }
    CUtensorMap mq, mg, mdl, ma;
    if (!make_tile_map(&mq, p.q, es, p.B, p.H, p.W, C, ch, 10, 6) || !make_tile_map(&mg, ga.dout, es, p.B, p.H, p.W, C, ch, 10, 6) ||
        !make_tile_map(&mdl, ws.rows_dl, 2, p.B, p.H, p.W, C, 32, 10, 6) || !make_tile_map(&ma, ws.rows_a, 2, p.B, p.H, p.W, C, 32, 10, 6))
        return cudaErrorInvalidValue;
    if (ws.rows_dl == ga.dv) P.sides = 1;
    for (; P.first_side < 2 && e == cudaSuccess; P.first_side += P.sides)
        e = launch_chained(bwd_gather_kernel<T>, grid, kThreads, Plan<kGatherImages>::total, stream, mdl, ma, mq, mg, P);
    return e;
}

size_t rows_bytes(int B, int H, int W, int heads) { return (size_t)B * H * W * heads * 64; }

}  // namespace

size_t bwd_team_workspace_bytes(int B, int H, int W, int heads, bool compact) {
    return (compact ? 1 : 2) * (rows_bytes(B, H, W, heads) + 256) + (size_t)heads * kImages;
}

BwdScratch bwd_scratch(void* ws, bool compact, void* dv, int B, int H, int W, int heads) {
    const size_t rows = (rows_bytes(B, H, W, heads) + 255) & ~(size_t)255;
    BwdScratch s;
    s.rows_a = static_cast<unsigned char*>(ws);
    s.rows_dl = compact ? static_cast<unsigned char*>(dv) : s.rows_a + rows;
    s.images = s.rows_a + (compact ? 1 : 2) * rows;
    return s;
}

cudaError_t launch_bwd_team(BwdPass what, const Problem& p, const BackwardArgs& ga, const BwdScratch& ws, int* d_status, int num_sms, cudaStream_t stream) {
    return p.dtype == SLIDE_ATTN_BF16 ? launch_t<__nv_bfloat16>(what, p, ga, ws, d_status, num_sms, stream) : launch_t<float>(what, p, ga, ws, d_status, num_sms, stream);
}

}  // namespace slide_attn
