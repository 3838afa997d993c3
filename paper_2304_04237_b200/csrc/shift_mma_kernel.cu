// Fixed-shift fast path for bf16 on tensor cores (head_dim 32): with the one-hot kernels of Eq. 11 slot s of a query
// pixel is the key / value at window offset s, so the forward is plain k x k local attention with zero padding,
//
//   l[s] = (q[p] . k[p + off(s)]) / sqrt(d) + bias[s]     a = softmax_s(l)     out[p,c] = sum_s a[s] v[p + off(s), c]
//
// as a banded attention in mma.sync.m16n8k16 tiles.  M = 16 queries = 2 rows x 8 columns; their windows cover k + 1 rows of 16
// keys, two n-tiles a row, of which k + 1 <= 10 columns of each row are inside a query's window; the logits of the others become
// -inf.  The logits' C fragments are the A fragments of
// the product with V.  The softmax weights go in as hi + lo (two bf16): the products of q and k are exact, V is exact, so
// the result has fp32 accuracy up to its own rounding, as the CUDA-core kernel has.
//
// The channels of q and k are taken in the order of a lane's 16-byte piece (any order will do for a dot product), so an
// operand of eight keys is one conflict-free 16-byte load per lane.  V comes in two planes of 16 channels (32 bytes a pixel),
// read by transposing ldmatrix; the result is transposed within quads of lanes to leave in 16-byte stores.
//
// One CTA = one head of a 4 x tw pixel tile (tw <= 32: with 56 columns, or 8 rows, fewer CTAs share an SM and cover each other's
// loads, 61 -> 65, 97 us at 64 x 56 x 56, 3 heads, k = 5), one warp per 8 columns; K and V tile + halo and the q tile by TMA
// (out-of-map elements zero-filled: that IS the padding).  Values up to seven columns outside a window enter the products with weight
// 0, and 0 times an infinity or a NaN would spread to queries that do not see it: a warp whose sums are not all finite takes them
// again, window by window (plain_rows; with the test k = 9 is 2 % slower).
//
// k = 5, 7, 9: with k = 3 nine tenths of the band are masked, and the CUDA-core kernel is faster (64 x 56 x 56, 3 heads: 36 us
// against 44).  A call (weight check and kernel) on CUDA cores and here, 64 x 56 x 56, 3 heads: k = 5 70 and 59 us, k = 7 124 and 75; 16 x
// 56 x 56, 3 heads, k = 9: 62 and 34 us.
#include "common.cuh"
#include "ptx.cuh"
#include "split.cuh"

namespace slide_attn {

namespace {

constexpr int kHeadDim = 32, kTH = 4, kMaxW = 32;
constexpr float kLog2e = 1.4426950408889634f;

struct ShiftMmaParams {
    const float* bias;
    __nv_bfloat16* out;
    int* status;
    int H, W, heads;
    int tw, tiles_x, tiles_y;
    float scale_log2e;
};

template <int K>
struct Plan {
    static constexpr int HH = kTH + K - 1;
    uint32_t v_off, v_plane, q_off, bar_off, total, tx_bytes;
    __host__ __device__ explicit Plan(int tw) {
        const uint32_t keys = (uint32_t)(HH * (tw + 8));
        auto up = [](uint32_t x) { return (x + 127u) & ~127u; };
        v_off = up(keys * 64u);
        v_plane = up(keys * 32u);
        q_off = v_off + 2 * v_plane;
        bar_off = q_off + up((uint32_t)(kTH * tw) * 64u);
        total = bar_off + 16 + 128;
        tx_bytes = keys * 128u + (uint32_t)(kTH * tw) * 64u;
    }
};

// The queries of the lane's column in rows r0 and r0 + 1 of the tile over their own windows only, in fp32.  `keys`, `values`, `queries`: the
// lane's 16-byte piece at the first pixel of its column; row pitches in bytes.
template <int K>
__device__ __noinline__ void plain_rows(const unsigned char* keys, const unsigned char* values, const unsigned char* queries, uint32_t key_pitch,
                                        uint32_t query_pitch, const float* bias, float scale_log2e, __nv_bfloat16* out, size_t out_pitch, int rows)
{
    auto widen = [](const unsigned char* p, float (&f)[8]) {
        const uint4 v = *reinterpret_cast<const uint4*>(p);
        f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x); f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
        f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z); f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
    };
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
        float q[8], acc[8], m = -INFINITY, z = 0.f;
        widen(queries + (uint32_t)r * query_pitch, q);
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = 0.f;
        auto logit = [&](int u, int v) {
            float k[8], l = 0.f;
            widen(keys + (uint32_t)(r + u) * key_pitch + (uint32_t)v * 64u, k);
#pragma unroll
            for (int c = 0; c < 8; ++c) l = fmaf(q[c], k[c], l);
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            return fmaf(l, scale_log2e, bias ? bias[u * K + v] * kLog2e : 0.f);
        };
#pragma unroll 1
        for (int u = 0; u < K; ++u)
#pragma unroll 1
            for (int v = 0; v < K; ++v) m = fmaxf(m, logit(u, v));
#pragma unroll 1
        for (int u = 0; u < K; ++u)
#pragma unroll 1
            for (int v = 0; v < K; ++v) {
                const float p = fast_exp2(logit(u, v) - m);
                float f[8];
                widen(values + (uint32_t)(r + u) * (key_pitch >> 1) + (uint32_t)v * 32u, f);
                z += p;
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[c] = fmaf(p, f[c], acc[c]);
            }
        const float inv = 1.f / z;
        if (r < rows)
            *reinterpret_cast<uint4*>(out + (size_t)r * out_pitch) = make_uint4(pack_bf16(acc[0] * inv, acc[1] * inv), pack_bf16(acc[2] * inv, acc[3] * inv),
                                                                                pack_bf16(acc[4] * inv, acc[5] * inv), pack_bf16(acc[6] * inv, acc[7] * inv));
    }
}

template <int K>
__global__ void __launch_bounds__(kMaxW * 4, K <= 5 ? 4 : 3)
shift_mma_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const ShiftMmaParams P)
{
    constexpr int R = K / 2;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    const Plan<K> L(P.tw);
    const uint32_t bar = smem_u32(smem) + L.bar_off;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, tig = lane & 3;
    const int h = blockIdx.x % P.heads;
    int tile = blockIdx.x / P.heads;
    const int tx = tile % P.tiles_x; tile /= P.tiles_x;
    const int ty = tile % P.tiles_y;
    const int b = tile / P.tiles_y;
    const int x0 = tx * P.tw, y0 = ty * kTH, HW = P.tw + 8;

    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, L.tx_bytes);
        const int c0 = h * kHeadDim;
        tma_load_4d(smem_u32(smem), &map_k, bar, c0, x0 - R, y0 - R, b);
        tma_load_4d(smem_u32(smem) + L.q_off, &map_q, bar, c0, x0, y0, b);
        tma_load_4d(smem_u32(smem) + L.v_off, &map_v, bar, c0, x0 - R, y0 - R, b);
        tma_load_4d(smem_u32(smem) + L.v_off + L.v_plane, &map_v, bar, c0 + 16, x0 - R, y0 - R, b);
    }
    // column n = 8 j + 2 tig + e of a row of keys is window column v = n - g of the lane's queries
    float tab[K][4];
    bool in[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int v = 8 * (i >> 1) + 2 * tig + (i & 1) - g;
        in[i] = v >= 0 && v < K;
#pragma unroll
        for (int u = 0; u < K; ++u) tab[u][i] = in[i] && P.bias ? P.bias[(h * K + u) * K + v] * kLog2e : 0.f;
    }
    __syncthreads();
    if (!mbar_wait(bar, 0)) {                                        // bounded
        if (lane == 0) atomicExch(P.status, 1);
        if (threadIdx.x == 0) grid_dependency_wait();
        return;
    }

    const unsigned char* keys = smem + (uint32_t)(8 * warp + g) * 64u + (uint32_t)tig * 16u;
    const uint32_t values = smem_u32(smem) + L.v_off + (uint32_t)(8 * warp + (lane & 15)) * 32u + (uint32_t)(lane >> 4) * 16u;
    const unsigned char* queries = smem + L.q_off + (uint32_t)(8 * warp + g) * 64u + (uint32_t)tig * 16u;
    const int C = P.heads * kHeadDim, x = x0 + 8 * warp + g;
#pragma unroll 1
    for (int r0 = 0; r0 < kTH && y0 + r0 < P.H; r0 += 2) {
        const uint4 qa = *reinterpret_cast<const uint4*>(queries + (uint32_t)(r0 * P.tw) * 64u);
        const uint4 qb = *reinterpret_cast<const uint4*>(queries + (uint32_t)((r0 + 1) * P.tw) * 64u);
        const uint32_t a0[4] = {qa.x, qb.x, qa.y, qb.y}, a1[4] = {qa.z, qb.z, qa.w, qb.w};
        float s[K + 1][2][4];
#pragma unroll
        for (int hr = 0; hr <= K; ++hr)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint4 kv = *reinterpret_cast<const uint4*>(keys + (uint32_t)((r0 + hr) * HW + 8 * j) * 64u);
                mma_bf16_c(s[hr][j], a0, kv.x, kv.y, 0.f, 0.f, 0.f, 0.f);
                mma_bf16(s[hr][j], a1, kv.z, kv.w);
            }
        // query row 0 (elements 0, 1) has the key rows 0 .. K - 1, query row 1 (2, 3) the rows 1 .. K
        float inv[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float m = -INFINITY, z = 0.f;
#pragma unroll
            for (int u = 0; u < K; ++u)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float& v = s[u + q][i >> 1][2 * q + (i & 1)];
                    v = in[i] ? fmaf(v, P.scale_log2e, tab[u][i]) : -INFINITY;
                    m = fmaxf(m, v);
                }
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
#pragma unroll
            for (int u = 0; u < K; ++u)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float& v = s[u + q][i >> 1][2 * q + (i & 1)];
                    v = fast_exp2(v - m);
                    z += v;
                }
            z += __shfl_xor_sync(0xffffffffu, z, 1);
            z += __shfl_xor_sync(0xffffffffu, z, 2);
            inv[q] = 1.f / z;
            const int none = q == 0 ? K : 0;                         // the row of keys that is not this query row's
#pragma unroll
            for (int j = 0; j < 2; ++j) { s[none][j][2 * q] = 0.f; s[none][j][2 * q + 1] = 0.f; }
        }
        float o[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) o[c][i] = 0.f;
#pragma unroll
        for (int hr = 0; hr <= K; ++hr) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {                            // a0, a1: keys 0 - 7 of query rows 0, 1; a2, a3: keys 8 - 15
                const float p0 = s[hr][i >> 1][2 * (i & 1)], p1 = s[hr][i >> 1][2 * (i & 1) + 1];
                hi[i] = pack_bf16(p0, p1);
                lo[i] = pack_bf16(p0 - bf16_lo(hi[i]), p1 - bf16_hi(hi[i]));
            }
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                uint32_t v[4];
                split::ldmatrix_x4_trans(values + (uint32_t)p * L.v_plane + (uint32_t)((r0 + hr) * HW) * 32u, v[0], v[1], v[2], v[3]);
                mma_bf16(o[2 * p], hi, v[0], v[1]);
                mma_bf16(o[2 * p + 1], hi, v[2], v[3]);
                mma_bf16(o[2 * p], lo, v[0], v[1]);
                mma_bf16(o[2 * p + 1], lo, v[2], v[3]);
            }
        }
        float finite = 0.f, unused = 0.f;                            // 0 times a sum: 0 unless one is not finite
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            ffma2(finite, unused, o[c][0], o[c][1], 0.f, 0.f);
            ffma2(finite, unused, o[c][2], o[c][3], 0.f, 0.f);
        }
        if (__any_sync(0xffffffffu, !(finite + unused == 0.f))) {
            const int y = y0 + r0;
            plain_rows<K>(keys + (uint32_t)(r0 * HW) * 64u,
                          smem + L.v_off + (uint32_t)(tig >> 1) * L.v_plane + (uint32_t)(r0 * HW + 8 * warp + g) * 32u + (uint32_t)(tig & 1) * 16u,
                          queries + (uint32_t)(r0 * P.tw) * 64u, (uint32_t)HW * 64u, (uint32_t)P.tw * 64u, P.bias ? P.bias + h * K * K : nullptr, P.scale_log2e,
                          P.out + ((size_t)(b * P.H + y) * P.W + x) * C + h * kHeadDim + tig * 8, (size_t)P.W * C, x < P.W ? (y + 1 < P.H ? 2 : 1) : 0);
            continue;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t w[4];                                           // word c: channels 8 c + 2 tig, + 1
#pragma unroll
            for (int c = 0; c < 4; ++c) w[c] = pack_bf16(o[c][2 * q] * inv[q], o[c][2 * q + 1] * inv[q]);
            // 4 x 4 transpose in the quad: word c of lane t becomes word t of lane c
            const bool b0 = tig & 1, b1 = tig & 2;
#pragma unroll
            for (int c = 0; c < 4; c += 2) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, b0 ? w[c] : w[c + 1], 1);
                if (b0) w[c] = got; else w[c + 1] = got;
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, b1 ? w[c] : w[c + 2], 2);
                if (b1) w[c] = got; else w[c + 2] = got;
            }
            const int y = y0 + r0 + q;
            if (x < P.W && y < P.H)
                *reinterpret_cast<uint4*>(P.out + ((size_t)(b * P.H + y) * P.W + x) * C + h * kHeadDim + tig * 8) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    if (threadIdx.x == 0) grid_dependency_wait();                    // not complete before the weight check (see launch_chained)
}

template <int K>
cudaError_t launch_t(const Problem& p, int* d_status, cudaStream_t stream) {
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !configured[dev]) {
        e = cudaFuncSetAttribute(shift_mma_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Plan<K>(kMaxW).total);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured[dev] = true;
    }
    // the tile width (a multiple of 8) that covers the map with the fewest columns, the widest of those
    int tw = 8, cover = 1 << 30;
    for (int t = 8; t <= kMaxW; t += 8) {
        const int c = (p.W + t - 1) / t * t;
        if (c <= cover) { cover = c; tw = t; }
    }
    ShiftMmaParams P;
    P.bias = p.bias; P.out = static_cast<__nv_bfloat16*>(p.out); P.status = d_status;
    P.H = p.H; P.W = p.W; P.heads = p.heads;
    P.tw = tw; P.tiles_x = (p.W + tw - 1) / tw; P.tiles_y = (p.H + kTH - 1) / kTH;
    P.scale_log2e = kLog2e / sqrtf((float)kHeadDim);
    const int C = p.heads * kHeadDim;
    CUtensorMap mq, mk, mv;
    if (!make_tile_map(&mq, p.q, 2, p.B, p.H, p.W, C, kHeadDim, tw, kTH) ||
        !make_tile_map(&mk, p.k, 2, p.B, p.H, p.W, C, kHeadDim, tw + 8, Plan<K>::HH) ||
        !make_tile_map(&mv, p.v, 2, p.B, p.H, p.W, C, 16, tw + 8, Plan<K>::HH))
        return cudaErrorInvalidValue;
    const long long ctas = (long long)P.tiles_x * P.tiles_y * p.B * p.heads;
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    // beside the weight check launched just before it; both only ever set the status word
    return launch_chained(shift_mma_kernel<K>, dim3((unsigned)ctas), tw * 4, Plan<K>(tw).total, stream, mq, mk, mv, P);
}

}  // namespace

cudaError_t launch_shift_mma(const Problem& p, int* d_status, cudaStream_t stream) {
    switch (p.ksize) {
        case 5: return launch_t<5>(p, d_status, stream);
        case 7: return launch_t<7>(p, d_status, stream);
        case 9: return launch_t<9>(p, d_status, stream);
        default: return cudaErrorInvalidConfiguration;
    }
}

}  // namespace slide_attn
