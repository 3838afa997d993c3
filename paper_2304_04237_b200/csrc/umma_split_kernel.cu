// UMMA_SPLIT variant (k = 3; fp32 storage or bf16; head_dim 16, 32 or 64): the fused forward (Eq. 2 with Eq. 12 inside)
// with fp32 arithmetic, both k^4 contractions on tcgen05.  Where UMMA_TS rounds the q.k products and the softmax
// weights to bf16, this kernel splits them, and the weights, into parts whose tensor-core products are exact
// (split.cuh, team.cuh).  Error against 64 bits (2-norm, fp32 storage, 4 x 56 x 56, 3 heads of 16, 3 of 32, 2 of 64): 1.22, 1.21,
// 1.22e-7, with q four times as large 1.29, 1.28, 1.30e-7; kernels of fp32 FMAs 1.29, 1.51, 1.30e-7 and 1.76, 2.24, 1.80e-7.
//
//   logits   l[s] = scale * sum_{t,c} (q[c] k_t[c]) wk[c,s,t] + bias[s]     a = softmax(l)
//   values   out[c] = sum_t v_t[c] (sum_s a[s] wv[c,s,t])
//
// Persistent, one CTA per SM, CTA c -> head c mod heads; two teams (team.cuh), each with a block of four strips at a time,
// blocks dealt over teams round-robin, neighbouring CTAs on neighbouring blocks.  A block's K planes, then its V planes
// come through the team's ring.
//
// Bound by latency: the chain products -> MMA -> softmax -> split rows -> MMA -> sum and its hand-offs, with four compute warps per
// scheduler to cover it.  Issue slots 30 - 36 % busy at 1.8 GHz, tensor pipe 13 - 24 %, DRAM 14 - 18 %.  A call, before (the CUDA-core kernel that
// took the shape) and here: 2 x 128 x 128, 3 heads, fp32: 45.2 us in tile_kernel, 28.9; 32 x 28 x 28, 3 heads of 64, bf16: 232 us in
// strip_kernel, 23.7; 1 x 14 x 14, 1 head, fp32: 14.4 and 7.5 - 8.1 us; heads of 16 (an earlier form of this kernel against strip_kernel): 16 x 56 x 56
// x 3, bf16 197 and 16.1, fp32 184 and 22.7 us.
#include "team.cuh"

namespace slide_attn {

namespace {

using namespace team;

template <typename T, int D>
struct Fwd {
    static constexpr int planes = D / Cut<T>::channels;
    static constexpr int chunks = 3 * planes;                                    // product chunks, and D chunks, of a block
    static constexpr uint32_t image = contract_bytes(D) + expand_bytes(D);      // of a head, in shared memory and in the workspace
    static constexpr uint32_t misc = 8u * (kTeams * kTeamBars + 1) + 16 + 16;       // barriers, tensor-memory slot; largest weight, another barrier
    static constexpr int fit = (int)((227u * 1024u - image - misc - 128) / (kTeams * kSlot));
    static constexpr int ring = fit < kMaxRing ? fit : kMaxRing;                 // slots of a team
    static_assert(ring >= 2, "the ring does not fit");
    // fp32 weights of a head, either side: they wait in the last slots of a team's ring, which the team does not need before
    static constexpr uint32_t raw = (uint32_t)D * kK2 * kK2 * 4;
    static constexpr int raw_slots = (int)((raw + kSlot - 1) / kSlot);
    static_assert(raw_slots < ring, "fp32 weights");
    static constexpr uint32_t raw_off = (uint32_t)((ring - raw_slots) * kSlot), raw_off_v = raw_off + (uint32_t)(ring * kSlot);
    static constexpr uint32_t w_off = (uint32_t)(kTeams * ring * kSlot);
    static constexpr uint32_t bar_off = w_off + ((image + 15u) & ~15u);
    static constexpr uint32_t total = bar_off + misc + 128;
};

struct SplitParams {
    const unsigned char* img;        // [head] contraction image of wk, expansion image of wv; null: built here
    const void* q;
    const float* bias;
    void* out;
    int* status;
    int H, W, heads;
    Strips strips;
    float scale_log2e;
    const float* wk;
    const float* wv;
};

template <typename T, int D>
__global__ void __launch_bounds__(256)
umma_split_prep_kernel(const float* __restrict__ wk, const float* __restrict__ wv, unsigned char* __restrict__ img)
{
    grid_dependency_wait();
    grid_launch_dependents();        // the main kernel may start its own prologue now
    const size_t w = (size_t)blockIdx.x * D * kK2 * kK2;
    unsigned char* dst = img + (size_t)blockIdx.x * Fwd<T, D>::image;
    build_images<T>(wk + w, dst, wv + w, dst + contract_bytes(D), D, blockIdx.y);
}

// Build: the CTAs lay out their head's weights themselves (see umma_split_builds_images; a kernel of its own, because the code for it costs
// others 5 % of a call, 2 x 128 x 128, 3 heads, fp32 28.6 us -> 30.0).
template <typename T, int D, bool Build>
__global__ void __launch_bounds__(kThreads, 1)
umma_split_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const SplitParams P)
{
    using F = Fwd<T, D>;
    using Piece = typename Cut<T>::piece;
    constexpr int NPL = F::planes, CH = Cut<T>::channels, PL = Cut<T>::per_lane, DB = Cut<T>::d_buffers, R = F::ring;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const uint32_t bars = smem_u32(smem + F::bar_off);
    const uint32_t bar_weights = bars + 8u * (kTeams * kTeamBars);
    unsigned char* tmem_slot = smem + F::bar_off + 8u * (kTeams * kTeamBars + 1);
    const uint32_t bar_raw = smem_u32(tmem_slot) + 16u;
    uint32_t* s_most = reinterpret_cast<uint32_t*>(tmem_slot + 24);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int h = blockIdx.x % P.heads, rank = blockIdx.x / P.heads, nrank = (int)gridDim.x / P.heads;
    const int team_id = warp < kComputeWarps ? warp / kTeamWarps : (warp - kComputeWarps) % kTeams;
    const int blocks = (int)((P.strips.total + 3) >> 2);
    const int first = team_id * nrank + rank, step = kTeams * nrank;
    const int my_blocks = first < blocks ? (blocks - first + step - 1) / step : 0;
    const uint32_t tb = bars + 8u * (uint32_t)(team_id * kTeamBars);
    auto bar = [&](int i) { return tb + 8u * (uint32_t)i; };

    if (threadIdx.x == 0) {
        for (int i = 0; i < kTeams; ++i) init_team_bars(bars + 8u * (uint32_t)(i * kTeamBars));
        mbar_init_only(bar_weights, Build ? kComputeWarps : 1);
        if (Build) { mbar_init_only(bar_raw, 1); *s_most = 0u; }
        mbar_init_fence();
    }
    if (warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = *reinterpret_cast<const volatile uint32_t*>(tmem_slot) + kCols * (uint32_t)team_id;
    unsigned char* ring = smem + (uint32_t)(team_id * R * kSlot);
    bool ok = true;

    if (warp >= kTmaWarp) {
        // ---- TMA thread of a team: the K planes, then the V planes of every block -------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            int slot = 0, loads = 0;
            uint32_t phase = 1;                                      // a fresh barrier is free
            StripWalk at(P.strips, 4LL * first, 4LL * step);
            if (Build) grid_dependency_wait();                       // else the prep kernel has waited before it let this one start
            for (int bi = 0; ok && bi < my_blocks; ++bi, at.next()) {
                for (int v = 0; v < 2 * NPL; ++v) {
                    if (Build && loads++ == R - F::raw_slots && !mbar_wait(bar_weights, 0)) { ok = false; break; }       // the fp32 weights make room
                    if (!mbar_wait(bar(kEmpty + slot), phase)) { ok = false; break; }
                    const CUtensorMap* map = v < NPL ? &map_k : &map_v;
                    const int c0 = h * D + (v < NPL ? v : v - NPL) * CH;
                    load_strips(smem_u32(ring) + (uint32_t)(slot * kSlot), map, bar(kFull + slot), c0, at);
                    if (++slot == R) { slot = 0; phase ^= 1u; }
                }
            }
            // What follows in the stream may be launched: as blocks leave, it takes their place and sets itself up.
            if (Build && team_id == 0) grid_launch_dependents();
            if (!ok) atomicExch(P.status, 1);
        }
        __syncwarp();
    } else if (warp >= kMmaWarp) {
        // ---- MMA thread of a team -------------------------------------------------------------------
        uint32_t leader;
        if (elect_one(leader)) {
            if (warp == kMmaWarp) {                                  // the head's weights, once per CTA
                grid_dependency_wait();
                if constexpr (!Build) {
                    mbar_expect_tx(bar_weights, F::image);
                    bulk_load_1d(smem_u32(smem + F::w_off), P.img + (size_t)h * F::image, F::image, bar_weights);
                } else {
                    constexpr size_t floats = F::raw / 4;
                    mbar_expect_tx(bar_raw, 2 * F::raw);
                    bulk_load_1d(smem_u32(smem + F::raw_off), P.wk + h * floats, F::raw, bar_raw);
                    bulk_load_1d(smem_u32(smem + F::raw_off_v), P.wv + h * floats, F::raw, bar_raw);
                }
            }
            if (my_blocks > 0) ok = mbar_wait(bar_weights, 0);
            const uint64_t kdesc = contract_desc(smem_u32(smem + F::w_off));
            const uint32_t dsrc = smem_u32(smem + F::w_off) + contract_bytes(D);
            int pn = 0, dn = 0;                                      // chunks issued so far
            for (int bi = 0; ok && bi < my_blocks; ++bi) {
                for (int i = 0; i < F::chunks; ++i, ++pn) {          // plane, tap column
                    const int pb = pn & 1, plane = i / 3, dx = i % 3;
                    if (!mbar_wait(bar(kPFull + pb), (uint32_t)(pn >> 1) & 1u)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t p_col = tmem + kColP + (uint32_t)(pb * 3 * Cut<T>::tap_cols);
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy)
                        issue_contract<T>(tmem, p_col + dy * Cut<T>::tap_cols, kdesc + contract_step<T>(plane, dy * 3 + dx), plane, dx, dy);
                    umma_commit(bar(kPFree + pb));
                }
                if (!ok) break;
                umma_commit(bar(kLFull));
                if (!mbar_wait(bar(kAFull), (uint32_t)bi & 1u)) { ok = false; break; }
                for (int i = 0; i < F::chunks; ++i, ++dn) {
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
        const int w = warp % kTeamWarps, wq = w & 3, half = w >> 2, g = lane >> 2, tig = lane & 3;
        const uint32_t quad = tmem + ((uint32_t)(32 * wq) << 16), mine = quad + ((uint32_t)(16 * half) << 16);
        const int C = P.heads * D;
        if constexpr (Build) {                                       // the head's images, by the compute warps of both teams
            grid_dependency_wait();
            ok = warp_wait(bar_raw, 0);
            const float* raw = reinterpret_cast<const float*>(smem + F::raw_off);
            const float* raw_v = reinterpret_cast<const float*>(smem + F::raw_off_v);
            float most = 0.f;
            if constexpr (sizeof(T) == 4) {
                uint32_t m = 0;
                for (int i = threadIdx.x; i < (int)F::raw / 16; i += kComputeWarps * 32) {
                    const uint4 v = reinterpret_cast<const uint4*>(raw)[i];
                    m = max(max(m, max(v.x & 0x7fffffffu, v.y & 0x7fffffffu)), max(v.z & 0x7fffffffu, v.w & 0x7fffffffu));
                }
                m = __reduce_max_sync(0xffffffffu, m);
                if (lane == 0) atomicMax(s_most, m);
                asm volatile("bar.sync 1, %0;" ::"n"(kComputeWarps * 32) : "memory");
                most = __uint_as_float(*reinterpret_cast<volatile uint32_t*>(s_most));
            }
            unsigned char* img = smem + F::w_off;
            for (int i = threadIdx.x; i < contract_slots(D); i += kComputeWarps * 32) build_contract_slot<T>(raw, img, i, most);
            // from the other end, so that a thread has as few items of both kinds as can be
            for (int i = kComputeWarps * 32 - 1 - (int)threadIdx.x; i < D * kK2; i += kComputeWarps * 32)
                build_expand_item<T>(raw_v, img + contract_bytes(D), i);
            fence_proxy_async_smem();                                // the tensor core reads these bytes through the async proxy
            __syncwarp();
            mbar_arrive_lane0(bar_weights, lane);
        }
        float bias[kK2];
#pragma unroll
        for (int s = 0; s < kK2; ++s) bias[s] = P.bias ? P.bias[h * kK2 + s] * kLog2e : 0.f;

        int slot = 0, pn = 0, dn = 0;
        uint32_t phase = 0;
        const uint32_t zero = (uint32_t)(P.H >> 31);
        auto release = [&]() {                                       // the plane at `slot` has been read
            __syncwarp();
            mbar_arrive_lane0(bar(kEmpty + slot), lane);
            if (++slot == R) { slot = 0; phase ^= 1u; }
        };
        auto release_after = [&](float a, float b) {                // the sums a and b hold what was read from it
            __syncwarp();
            mbar_arrive_lane0_after(bar(kEmpty + slot), lane, a, b, zero);
            if (++slot == R) { slot = 0; phase ^= 1u; }
        };
        // the lane's first pixel: element offset of its piece, and which of its two rows are inside (past the last strip: none)
        const size_t row_pitch = (size_t)P.W * C;
        StripWalk walk(P.strips, 4LL * first + wq, 4LL * step);
        struct Place { size_t at; bool in[2]; };
        auto place = [&](int bi) {
            Place p;
            const int y = walk.y0() + 2 * half, x = walk.x0() + g;
            const bool in = 4LL * (first + (long long)bi * step) + wq < P.strips.total && x < P.W;
            p.in[0] = in && y < P.H; p.in[1] = in && y + 1 < P.H;
            p.at = (((size_t)walk.b * P.H + y) * P.W + x) * C + h * D + tig * PL;
            return p;
        };
        auto load_q = [&](const Place& p, int plane, Piece (&x)[2]) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                x[r] = Piece();
                if (p.in[r]) x[r] = __ldg(reinterpret_cast<const Piece*>(static_cast<const T*>(P.q) + p.at + r * row_pitch + plane * CH));
            }
        };
        Place st = place(0);
        Piece qn[2];
        if (my_blocks > 0) load_q(st, 0, qn);
        for (int bi = 0; bi < my_blocks; ++bi) {
            // ---- products -------------------------------------------------------------------------
            for (int pl = 0; pl < NPL; ++pl) {
                Factor<T> x;
                x.set(qn);
                if (pl + 1 < NPL) load_q(st, pl + 1, qn);
                if (!warp_wait(bar(kFull + slot), phase)) { ok = false; break; }
                const unsigned char* plane = ring + (uint32_t)(slot * kSlot + wq * kHaloPlane);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx, ++pn) {
                    const int pb = pn & 1;
                    Piece y[4];
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
                }
                if (!ok) break;
                release();
            }
            if (!ok) break;
            const Place cur = st;
            if (bi + 1 < my_blocks) { walk.next(); st = place(bi + 1); load_q(st, 0, qn); }

            // ---- softmax: thread = pixel of the quadrant; the two warps of a quadrant take turns -------------
            if (half == (bi & 1)) {
                if (!warp_wait(bar(kLFull), (uint32_t)bi & 1u)) { ok = false; break; }
                tc_fence_after_sync();
                float a[kK2];
                load_contraction<T>(quad, a);
                const float iz = 1.f / softmax_terms(a, P.scale_log2e, bias);
#pragma unroll
                for (int s = 0; s < kK2; ++s) a[s] *= iz;
                uint32_t row[16];
                split_row(a, row);
                tmem_st_32x32b_x16(quad + kColA, row);
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                mbar_arrive_lane0(bar(kAFull), lane);
            }

            // ---- values ----------------------------------------------------------------------------
            for (int pl = 0; pl < NPL; ++pl) {
                float acc[2][PL];
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int c = 0; c < PL; ++c) acc[r][c] = 0.f;
                if (!warp_wait(bar(kFull + slot), phase)) { ok = false; break; }
                const unsigned char* plane = ring + (uint32_t)(slot * kSlot + wq * kHaloPlane);
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
                for (int r = 0; r < 2; ++r) {
                    if (!cur.in[r]) continue;
                    Piece o;
                    if constexpr (sizeof(T) == 2) {
                        o.x = pack_bf16(acc[r][0], acc[r][1]); o.y = pack_bf16(acc[r][2], acc[r][3]);
                        if constexpr (PL == 8) { o.z = pack_bf16(acc[r][4], acc[r][5]); o.w = pack_bf16(acc[r][6], acc[r][7]); }
                    } else {
                        o.x = __float_as_uint(acc[r][0]); o.y = __float_as_uint(acc[r][1]);
                        o.z = __float_as_uint(acc[r][2]); o.w = __float_as_uint(acc[r][3]);
                    }
                    *reinterpret_cast<Piece*>(static_cast<T*>(P.out) + cur.at + r * row_pitch + pl * CH) = o;
                }
            }
            if (!ok) break;
        }
        if (!ok && lane == 0) atomicExch(P.status, 1);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after_sync();
        tmem_dealloc(*reinterpret_cast<const volatile uint32_t*>(tmem_slot), 512);
    }
}

template <typename T, int D>
cudaError_t launch_t(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream) {
    using F = Fwd<T, D>;
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(umma_split_kernel<T, D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::total);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(umma_split_kernel<T, D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::total);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured[dev] = true;
    }
    SplitParams P;
    P.wk = p.wk; P.wv = p.wv; P.img = static_cast<const unsigned char*>(workspace); P.q = p.q; P.bias = p.bias; P.out = p.out; P.status = d_status;
    P.H = p.H; P.W = p.W; P.heads = p.heads;
    P.strips.sx = (p.W + 7) / 8; P.strips.bands = (p.H + 3) / 4;
    P.strips.total = (long long)p.B * P.strips.bands * P.strips.sx;
    if (P.strips.total > 0x7fffffffLL - 4) return cudaErrorInvalidConfiguration;
    P.scale_log2e = kLog2e / sqrtf((float)D);
    CUtensorMap mk, mv;
    const int C = p.heads * D;
    if (!make_tile_map(&mk, p.k, (int)sizeof(T), p.B, p.H, p.W, C, Cut<T>::box, 10, 6) ||
        !make_tile_map(&mv, p.v, (int)sizeof(T), p.B, p.H, p.W, C, Cut<T>::box, 10, 6))
        return cudaErrorInvalidValue;
    const long long blocks = (P.strips.total + 3) / 4;
    long long per_head = num_sms / p.heads;
    if (per_head > blocks) per_head = blocks;
    if (per_head < 1) per_head = 1;
    return launch_chained(P.img ? umma_split_kernel<T, D, false> : umma_split_kernel<T, D, true>, dim3((unsigned)(per_head * p.heads)), kThreads, F::total, stream, mk, mv, P);
}

template <typename T, int D> struct Heads { using type = T; static constexpr int dim = D; };

// f(the instance of p's storage type and head width)
template <typename F>
cudaError_t of_heads(const Problem& p, F f) {
    if (p.dtype == SLIDE_ATTN_BF16) return p.head_dim == 16 ? f(Heads<NarrowBf16, 16>()) : p.head_dim == 32 ? f(Heads<__nv_bfloat16, 32>()) : f(Heads<__nv_bfloat16, 64>());
    return p.head_dim == 16 ? f(Heads<float, 16>()) : p.head_dim == 32 ? f(Heads<float, 32>()) : f(Heads<float, 64>());
}

}  // namespace

bool umma_split_supports(int head_dim, int ksize) {
    return (head_dim == 16 || head_dim == 32 || head_dim == 64) && ksize == 3 && tensor_map_available();
}

size_t umma_split_workspace_bytes(int heads, int head_dim) {
    return (size_t)heads * (contract_bytes(head_dim) + expand_bytes(head_dim));
}

// Whether the CTAs of the main launch lay out their head's weights themselves: where no team has more than one block.  Beside a prep
// launch a team starts on its first block 1 us earlier, as its warps are free for that, but the launch itself takes 2 us of a small call.
// With it / without, us: 1 x 14 x 14, 1 head, fp32 8.5 - 8.9 / 7.5 - 8.1; 4 x 28 x 28, 3 heads of 16, bf16 7.2 / 5.1; heads of 64, bf16, a block for
// every other SM 8.9 / 9.1, for every team 11.6 / 11.0.  Two blocks a team: 98 x 16 x 16, 3 heads, fp32 20.3 / 18.7, of 64, bf16 18.5 / 17.4, so the
// line could lie there; three: 2 x 128 x 128, 3 heads, fp32 28.6 / 29.0, 32 x 28 x 28, 3 heads of 64, bf16 23.6 / 24.2.
bool umma_split_builds_images(int B, int H, int W, int heads, int num_sms) {
    const long long blocks = ((long long)B * ((H + 3) / 4) * ((W + 7) / 8) + 3) / 4, per_head = num_sms / heads;
    return blocks <= kTeams * (per_head < 1 ? 1 : per_head);
}

// Weights -> images in `workspace`.
cudaError_t launch_umma_split_prep(const Problem& p, void* workspace, cudaStream_t stream) {
    return of_heads(p, [&](auto heads) {
        using H = decltype(heads);
        const dim3 grid((unsigned)p.heads, prep_parts(H::dim));
        unsigned char* img = static_cast<unsigned char*>(workspace);
        // Heads of 16 have little to lay out: spread, 17 x 48 x 51, 7 heads, bf16 takes 29.5 us instead of 29.2, and what follows UMMA_TS gains 2 % at most.
        if constexpr (H::dim > 16) return launch_spread<umma_split_prep_kernel<typename H::type, H::dim>>(grid, 256, stream, p.wk, p.wv, img);
        else return launch_chained(umma_split_prep_kernel<typename H::type, H::dim>, grid, 256, 0, stream, p.wk, p.wv, img);
    });
}

cudaError_t launch_umma_split(const Problem& p, const void* workspace, int* d_status, int num_sms, cudaStream_t stream) {
    return of_heads(p, [&](auto heads) {
        using H = decltype(heads);
        return launch_t<typename H::type, H::dim>(p, workspace, d_status, num_sms, stream);
    });
}

}  // namespace slide_attn
