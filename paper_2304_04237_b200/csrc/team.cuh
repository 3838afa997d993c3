// Shared by the kernels that run the split contractions on tcgen05 (exact products, fp32 accumulation; see
// split.cuh): geometry, the shared-memory images of the weights and the hand-offs of a team.
//
// A TEAM is eight warps with one block of 128 pixels (the 128 lanes of tensor memory) at a time; two teams share an SM
// and its weight images and run independently of each other, so that one team's hand-offs (180 - 220 cycles from an
// MMA's issue to the wake-up of its readers) are covered by the other's arithmetic.  (Four teams of four warps with
// one tap per hand-off, which leaves each team 128 columns, were 13 % slower with 64 channels a head.)
// A block is four STRIPS of 4 rows x 8 columns of the map; warps q and q + 4 of a team have quadrant q of tensor memory
// = strip q, the first its rows 0 and 1, the second rows 2 and 3: lane (g, tig) works on column g and piece tig of the
// channels of two rows, TMEM lane 32 q + 16 half + 8 row + g.  A strip is loaded by TMA with its halo (6 x 10 pixels,
// 64-byte channel planes, zero fill = the padding).  Four more warps: an MMA thread and a TMA thread per team.
//
//   products    x . y per (plane, tap column dx), split into parts, to tensor memory (a chunk; two buffers)
//   contraction L[p][n] += parts . Bk.  The columns of Bk are three groups of 16, nine used: the upper, middle and
//               lower part of the weight of each slot.  Upper x upper accumulates apart (H) from everything smaller (R);
//               they meet in registers.  The tensor core truncates whenever it adds to H, so:
//               bf16: three tiles H, one per tap column, whose sums stay small (two tiles, one per K step: error of the softmax
//               weights 1.9e-7, so: 1.4e-7, fp32 FMAs: 1.5e-7);
//               fp32: the upper parts are multiples of one power of two per pixel and plane (2^-8 of the largest product its window
//               can have), those of the weights of one per head, so that the sums in H are integers below 2^24 of their product:
//               exact.  (A product below that power of two keeps its 17 upper bits.)
//   softmax     one thread has a pixel's nine slots; the largest logit is subtracted before anything is rounded to scale
//   expansion   D[p][(tap, channel)] = A'[p][32] . Bv[64][(tap, channel)]: the three parts of the slot value against the three
//               parts of the weight, without the pairs below 2^-24 of the product
//   sum         sum_t D[p][t][c] y_t[p][c] with packed fp32 FMAs
//
// Tensor-memory columns of a team: product chunks, then 64 of sums (bf16: three H, R; fp32: H, R of 2^-8, 2^-16 and 2^-24 of
// it); later D in 0 - 191 and A' in the last 16.
#pragma once
#include "common.cuh"
#include "ptx.cuh"
#include "split.cuh"

namespace slide_attn {
namespace team {

constexpr int kTeams = 2, kTeamWarps = 8;
constexpr int kComputeWarps = kTeams * kTeamWarps;
constexpr int kMmaWarp = kComputeWarps, kTmaWarp = kMmaWarp + kTeams;          // one of each per team
constexpr int kThreads = (kTmaWarp + kTeams) * 32;
constexpr int kK2 = 9;
constexpr int kHaloPlane = 60 * 64;                     // bytes of one plane of a strip with its halo
constexpr int kSlot = 4 * kHaloPlane;                   // of a block: a slot of the team's ring
constexpr float kLog2e = 1.4426950408889634f;
constexpr uint32_t kCols = 256, kColP = 0, kColA = 240, kColD = 0;

// How the channels of a storage type are cut: planes of 64 bytes, chunks of one plane and one tap column.
template <typename T> struct Cut;
// bf16 storage with 16 channels a head.  Its planes keep the 64-byte pitch: TMA brings the next head's channels (past the
// last head: zeros) along, which nobody reads.
struct NarrowBf16 { __nv_bfloat16 v; };
template <> struct Cut<__nv_bfloat16> {
    using piece = uint4;                                // a lane's channels of a pixel
    static constexpr int channels = 32;                 // of a plane
    static constexpr int box = 32;                      // channels that a TMA box takes
    static constexpr int per_lane = 8;
    static constexpr int d_buffers = 2;                 // N = 96 columns per tap column of a plane
    static constexpr int tap_cols = 32;                 // products are hi + lo: 2 x 3 x 32 + 64 = 256 columns
};
template <> struct Cut<NarrowBf16> {
    using piece = uint2;
    static constexpr int channels = 16;
    static constexpr int box = 32;
    static constexpr int per_lane = 4;
    static constexpr int d_buffers = 3;                 // N = 48
    static constexpr int tap_cols = 16;                 // hi + lo: 2 x 3 x 16 + 64 = 160 columns
};
template <> struct Cut<float> {
    using piece = uint4;
    static constexpr int channels = 16;
    static constexpr int box = 16;
    static constexpr int per_lane = 4;
    static constexpr int d_buffers = 3;                 // N = 48
    static constexpr int tap_cols = 24;                 // hi + mid + lo: 2 x 3 x 24 + 64 = 208
};
template <typename T> constexpr uint32_t kColL = 6 * Cut<T>::tap_cols;          // the sums

// Channel of K index kappa within a plane (the order in which tcgen05.st lays the pieces out); the channel of column n of
// a tap of D (the order in which tcgen05.ld hands them to the lanes) is (CH / 4) ((n & 7) >> 1) + 2 (n >> 3) + (n & 1).
template <typename T> __host__ __device__ constexpr int channel_of_k(int kappa) {
    return Cut<T>::channels == 32 ? 8 * ((kappa & 15) >> 2) + (kappa & 3) + (kappa >= 16 ? 4 : 0) : kappa;
}

// Weight images of one head (bytes).  Contraction: [plane][tap][K / 8][48 n][8 k] bf16.  Expansion: [plane][tap
// column dx][dy][n][64 k] bf16 in core matrices.
__host__ __device__ constexpr uint32_t contract_bytes(int head_dim) { return (uint32_t)head_dim * 9u * 96u; }
__host__ __device__ constexpr uint32_t expand_bytes(int head_dim) { return (uint32_t)head_dim * 9u * 128u; }

// What rounds numbers up to `most` in magnitude to multiples of a power of two, so that the quotients are integers up to 256 and
// fit bf16: added and taken away again, 1.5 * 2^23 times that power.  Not for numbers from 2^112 on (`wide`), where it would be infinite.
__device__ __forceinline__ bool wide(float most) { return __float_as_uint(most) >= 0x77800000u; }       // NaN too
__device__ __forceinline__ float rounder(float most) { return __uint_as_float((__float_as_uint(most) & 0x7f800000u) + 0x08400000u); }

// The largest magnitude (a NaN counts as larger than anything) of each of N arrays of n floats, n a multiple of 4, by a block of 256.
template <int N>
__device__ __forceinline__ void block_most(const float* const (&w)[N], int n, float (&most)[N]) {
    __shared__ uint32_t s_most[N][8];
    uint32_t m[N] = {};
    for (int i = threadIdx.x; i < n / 4; i += 256)
#pragma unroll
        for (int a = 0; a < N; ++a) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(w[a]) + i);
            m[a] = max(max(m[a], max(v.x & 0x7fffffffu, v.y & 0x7fffffffu)), max(v.z & 0x7fffffffu, v.w & 0x7fffffffu));
        }
#pragma unroll
    for (int a = 0; a < N; ++a) {
        m[a] = __reduce_max_sync(0xffffffffu, m[a]);
        if ((threadIdx.x & 31) == 0) s_most[a][threadIdx.x >> 5] = m[a];
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < N; ++a) {
#pragma unroll
        for (int i = 0; i < 8; ++i) m[a] = max(m[a], s_most[a][i]);
        most[a] = __uint_as_float(m[a]);
    }
}

// Contraction image item: 16 bytes = 8 k of column n.  w: fp32 [head_dim][slot][tap] of the head.
template <typename T>
__device__ __forceinline__ void load_contract_item(const float* __restrict__ w, int item, float (&v)[8]) {
    constexpr int KG = Cut<T>::channels / 8;             // k groups of a (plane, tap)
    const int n = item % 48, kg = item / 48, s = n & 15;
    const int j = kg % KG, pt = kg / KG, tap = pt % kK2, plane = pt / kK2;
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = s < kK2 ? w[((plane * Cut<T>::channels + channel_of_k<T>(8 * j + e)) * kK2 + s) * kK2 + tap] : 0.f;
}
// `most` (fp32 storage): the largest of all weights of the head.
template <typename T>
__device__ __forceinline__ void build_contract_item(const float (&w)[8], unsigned char* img, int item, float most) {
    const int n = item % 48, kg = item / 48, part = n >> 4;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        v[e] = w[e];
        if (sizeof(T) == 4 && !wide(most)) {
            const float r = rounder(most), hi = __fadd_rn(__fadd_rn(v[e], r), -r), rest = v[e] - hi, mid = __bfloat162float(__float2bfloat16_rn(rest));
            v[e] = part == 0 ? hi : part == 1 ? mid : __bfloat162float(__float2bfloat16_rn(rest - mid));
        } else {
            if (part >= 1) v[e] = split::rest(v[e]);
            if (part >= 2) v[e] = split::rest(v[e]);
        }
    }
    *reinterpret_cast<uint4*>(img + (size_t)kg * 768 + (n >> 3) * 128 + (n & 7) * 16) =
        make_uint4(split::pack_upper(v[0], v[1]), split::pack_upper(v[2], v[3]), split::pack_upper(v[4], v[5]), split::pack_upper(v[6], v[7]));
}

// The same by slot: 8 k of one slot (of 16, nine used) for all three column groups, for few threads with many items.
__host__ __device__ constexpr int contract_slots(int head_dim) { return head_dim / 8 * kK2 * 16; }
template <typename T>
__device__ __forceinline__ void build_contract_slot(const float* w, unsigned char* img, int item, float most) {
    const int s = item & 15, kg = item >> 4;
    float x[8], v[3][8];
    load_contract_item<T>(w, kg * 48 + s, x);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        if (sizeof(T) == 4 && !wide(most)) {
            const float r = rounder(most), hi = __fadd_rn(__fadd_rn(x[e], r), -r), rest = x[e] - hi, mid = __bfloat162float(__float2bfloat16_rn(rest));
            v[0][e] = hi; v[1][e] = mid; v[2][e] = __bfloat162float(__float2bfloat16_rn(rest - mid));
        } else {
            v[0][e] = x[e]; v[1][e] = split::rest(x[e]); v[2][e] = split::rest(v[1][e]);
        }
    }
#pragma unroll
    for (int part = 0; part < 3; ++part) {
        const float (&p)[8] = v[part];
        *reinterpret_cast<uint4*>(img + kg * 768 + part * 256 + (s >> 3) * 128 + (s & 7) * 16) =
            make_uint4(split::pack_upper(p[0], p[1]), split::pack_upper(p[2], p[3]), split::pack_upper(p[4], p[5]), split::pack_upper(p[6], p[7]));
    }
}

// ---- the expansion's operands ----------------------------------------------------------------------------------------------
// Slot values (softmax weights, gradients) and weights have three bf16 parts each, so their magnitude does not matter.  (With
// two fp16 parts each, scaled to that type's range, a forward took half the MMAs and was not faster (2 x 128 x 128, 3 heads, fp32: 29.1 us,
// 26.7 here), and values above 2^100 overflowed before the scale was undone.)
// SPLIT ROW: 64 bytes of a pixel and head, 32 bf16: 0 - 8 upper parts of the slots, 9 - 17 middle, 18 - 26 lower parts, 27, 28
// the middle parts of slots 7 and 8 again.  In memory its four 16-byte pieces are swizzled by the pixel's column x (piece c
// at c ^ ((x >> 1) & 3)), which makes reads of eight neighbouring pixels' pieces free of bank conflicts.
// It meets an image of four 16-row K steps: rows 0 - 15 of the row with the upper parts of the weights, 16 - 31 likewise
// (27, 28 with the middle parts of slots 7 and 8), 0 - 15 with the middle parts, 0 - 8 with the lower parts: everything down to
// 2^-24 of the product.
// The lower parts carry what the tensor core's one truncation at full magnitude takes off a product on average: half a unit in the last
// place, relative to a number spread evenly over its logarithm 2^-24 / (2 ln 2).  (A single product of 8-bit numbers stays exact.)
constexpr float kTruncation = 4.3e-8f;
template <typename T>
__device__ __forceinline__ void build_expand_item(const float* __restrict__ w, unsigned char* img, int item) {
    constexpr int CH = Cut<T>::channels;
    const int n = item % CH, r = item / CH, dy = r % 3, dx = (r / 3) % 3, plane = r / 9;
    const int c = plane * CH + (CH / 4) * ((n & 7) >> 1) + 2 * (n >> 3) + (n & 1), tap = dy * 3 + dx;
    float hi[kK2], mid[kK2], lo[kK2];
#pragma unroll
    for (int s = 0; s < kK2; ++s) {
        hi[s] = w[(c * kK2 + s) * kK2 + tap];
        mid[s] = split::rest(hi[s]);
        lo[s] = __bfloat162float(__float2bfloat16_rn(fmaf(kTruncation, hi[s], split::rest(mid[s]))));
    }
    float v[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = 0.f;
#pragma unroll
    for (int s = 0; s < kK2; ++s) {
        v[s] = hi[s]; v[9 + s] = hi[s]; v[18 + s] = hi[s];
        v[32 + s] = mid[s]; v[48 + s] = lo[s];
    }
    v[27] = mid[7]; v[28] = mid[8];
#pragma unroll
    for (int s = 0; s < 7; ++s) v[41 + s] = mid[s];
    unsigned char* col = img + (size_t)(item >> 3) * 1024 + (item & 7) * 16;
#pragma unroll
    for (int j = 0; j < 8; ++j)
        *reinterpret_cast<uint4*>(col + j * 128) = make_uint4(split::pack_upper(v[8 * j], v[8 * j + 1]), split::pack_upper(v[8 * j + 2], v[8 * j + 3]),
                                                              split::pack_upper(v[8 * j + 4], v[8 * j + 5]), split::pack_upper(v[8 * j + 6], v[8 * j + 7]));
}
// The split row of nine slot values: 16 registers of two.
__device__ __forceinline__ void split_row(const float (&a)[kK2], uint32_t (&row)[16]) {
    float v[28];
#pragma unroll
    for (int s = 0; s < kK2; ++s) { v[s] = a[s]; v[9 + s] = split::rest(v[s]); v[18 + s] = split::rest(v[9 + s]); }
    v[27] = v[16];
#pragma unroll
    for (int i = 0; i < 14; ++i) row[i] = split::pack_upper(v[2 * i], v[2 * i + 1]);
    row[14] = split::pack_upper(v[17], 0.f);
    row[15] = 0u;
}
// The MMAs of N columns of D: B at `b_smem` (of the image), A = a split row in 16 columns at `a_col`.  The smallest products come
// first, so that the tensor core, which truncates whatever it adds to, truncates at full magnitude once.
template <int N>
__device__ __forceinline__ void issue_expand(uint32_t d_col, uint32_t a_col, uint32_t b_smem) {
    constexpr uint32_t idesc = umma_idesc_bf16(128, N);
    const uint64_t b = umma_smem_desc(b_smem, 128, 1024);                    // a K step further: 256 bytes = 16
    umma_bf16_ts(d_col, a_col, b + 48, idesc, 0);
    umma_bf16_ts(d_col, a_col + 8, b + 16, idesc, 1);
    umma_bf16_ts(d_col, a_col, b + 32, idesc, 1);
    umma_bf16_ts(d_col, a_col, b, idesc, 1);
}

// The images of one head by prep_parts(head_dim) blocks of 256 threads, of which this one is `part`: a thread per item of the
// expansion image, then of the contraction image.  (Four blocks a head took 12 us, most of what a small map needs.)
__host__ __device__ constexpr int expand_parts(int head_dim) { return (head_dim * kK2 + 255) / 256; }
__host__ __device__ constexpr int prep_parts(int head_dim) { return expand_parts(head_dim) + (head_dim / 8 * kK2 * 48 + 255) / 256; }
template <typename T>
__device__ __forceinline__ void build_images(const float* wc, unsigned char* cimg, const float* we, unsigned char* eimg, int head_dim, int part) {
    const int ce = part - expand_parts(head_dim), i = (ce < 0 ? part : ce) * 256 + threadIdx.x;
    if (ce < 0) {
        if (i < head_dim * kK2) build_expand_item<T>(we, eimg, i);
        return;
    }
    const bool in = i < head_dim / 8 * kK2 * 48;
    float w[8];
    if (in) load_contract_item<T>(wc, i, w);                                 // on their way while the largest weight is looked for
    float most[1] = {0.f};
    const float* const src[1] = {wc};
    if constexpr (sizeof(T) == 4) block_most<1>(src, head_dim * kK2 * kK2, most);
    if (in) build_contract_item<T>(w, cimg, i, most[0]);
}

// (A vote in every probe, which makes all branches of the wait uniform, measured 5 - 8 % slower than one at the end.)
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}

// Barriers of a team; kFull, kEmpty: its ring of planes.
constexpr int kMaxRing = 5;
enum : int { kPFull = 0, kPFree = 2, kLFull = 4, kAFull = 5, kDFull = 6, kDFree = 9, kFull = 12, kEmpty = kFull + kMaxRing,
             kLFree = kEmpty + kMaxRing, kTeamBars };

__device__ __forceinline__ void init_team_bars(uint32_t base) {
    auto init = [&](int i, uint32_t count) { mbar_init_only(base + 8u * (uint32_t)i, count); };
    for (int i = 0; i < 2; ++i) { init(kPFull + i, kTeamWarps); init(kPFree + i, 1); }
    init(kLFull, 1);
    init(kLFree, 4);
    init(kAFull, 4);
    for (int i = 0; i < 3; ++i) { init(kDFull + i, 1); init(kDFree + i, kTeamWarps); }
    for (int i = 0; i < kMaxRing; ++i) { init(kFull + i, 1); init(kEmpty + i, kTeamWarps); }
}

// Which strip of 4 rows x 8 columns: a walk over the strips of the maps from a given one in equal steps, without a
// division per step (dx, dy, db: the step as a number in the mixed base of columns, rows and images).
struct Strips {
    int sx, bands;
    long long total;                                     // B * bands * sx
};
struct StripWalk {
    int b, y, x;                                         // in strips; the strip's first pixel is (4 y, 8 x)
    int db, dy, dx, sx, bands;
    __device__ __forceinline__ StripWalk(const Strips& s, long long first, long long step) : sx(s.sx), bands(s.bands) {
        const int i = (int)first, d = (int)step;
        x = i % sx; y = i / sx % bands; b = i / sx / bands;
        dx = d % sx; dy = d / sx % bands; db = d / sx / bands;
    }
    __device__ __forceinline__ void next() {
        x += dx; y += dy; b += db;
        if (x >= sx) { x -= sx; ++y; }
        if (y >= bands) { y -= bands; ++b; }
    }
    __device__ __forceinline__ int x0() const { return 8 * x; }
    __device__ __forceinline__ int y0() const { return 4 * y; }
};

// One slot of a ring: arms the barrier and sends for a plane of the block's four strips, the first of them at `at` (strips
// past the last one read as zero: their image does not exist).
__device__ __forceinline__ void load_strips(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, StripWalk at) {
    mbar_expect_tx(bar, kSlot);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        tma_load_4d(dst + (uint32_t)(i * kHaloPlane), map, bar, c0, at.x0() - 1, at.y0() - 1, at.b);
        if (++at.x == at.sx) { at.x = 0; if (++at.y == at.bands) { at.y = 0; ++at.b; } }
    }
}

// Piece tig at pixel (row, column) of a halo plane.
template <typename T>
__device__ __forceinline__ typename Cut<T>::piece halo_piece(const unsigned char* plane, int row, int col, int tig) {
    using Piece = typename Cut<T>::piece;
    return *reinterpret_cast<const Piece*>(plane + (uint32_t)(row * 10 + col) * 64u + (uint32_t)tig * (uint32_t)sizeof(Piece));
}
__device__ __forceinline__ float f4(const uint4& v, int i) {
    return __uint_as_float(i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w);
}

// A lane's two left factors of the products.  bf16 keeps their negatives too: hi = x y and -lo = -x y + hi then need no
// negation in between, and the tensor core negates the low part (it was one instruction in seven of the products).
template <typename T> struct Factor;
template <> struct Factor<__nv_bfloat16> {
    uint4 x[2], nx[2];
    __device__ __forceinline__ void set(const uint4 (&v)[2]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            x[r] = v[r];
            nx[r] = make_uint4(v[r].x ^ 0x80008000u, v[r].y ^ 0x80008000u, v[r].z ^ 0x80008000u, v[r].w ^ 0x80008000u);
        }
    }
    __device__ __forceinline__ void meet(const unsigned char*, int, int, int, const uint4 (&)[4]) {}
};
template <> struct Factor<NarrowBf16> {
    uint2 x[2], nx[2];
    __device__ __forceinline__ void set(const uint2 (&v)[2]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) { x[r] = v[r]; nx[r] = make_uint2(v[r].x ^ 0x80008000u, v[r].y ^ 0x80008000u); }
    }
    __device__ __forceinline__ void meet(const unsigned char*, int, int, int, const uint2 (&)[4]) {}
};
// fp32 keeps what rounds the products of each pixel to their common power of two.
__device__ __forceinline__ float largest(const uint4& v) {
    return fmaxf(fmaxf(fabsf(f4(v, 0)), fabsf(f4(v, 1))), fmaxf(fabsf(f4(v, 2)), fabsf(f4(v, 3))));
}
template <> struct Factor<float> {
    uint4 x[2];
    float r[2];
    bool any_wide;
    __device__ __forceinline__ void set(const uint4 (&v)[2]) { x[0] = v[0]; x[1] = v[1]; }
    // what x will be multiplied with: the halo plane's rows `row` .. + 3, columns `col` (given: y0) .. + 2
    __device__ __forceinline__ void meet(const unsigned char* plane, int row, int col, int tig, const uint4 (&y0)[4]) {
        float y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            y[i] = largest(y0[i]);
#pragma unroll
            for (int dx = 1; dx < 3; ++dx) y[i] = fmaxf(y[i], largest(halo_piece<float>(plane, row + i, col + dx, tig)));
        }
        const float both = fmaxf(y[1], y[2]);
        float most[2] = {fmaxf(both, y[0]) * largest(x[0]), fmaxf(both, y[3]) * largest(x[1])};
        bool w = false;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            most[i] = fmaxf(most[i], __shfl_xor_sync(0xffffffffu, most[i], 1));
            most[i] = fmaxf(most[i], __shfl_xor_sync(0xffffffffu, most[i], 2));
            w = w || wide(most[i]);
            r[i] = rounder(most[i]);
        }
        any_wide = __any_sync(0xffffffffu, w);
    }
};
// Products of one tap of a plane for the lane's two pixels, split, into tensor memory at column `t`.
__device__ __forceinline__ void store_products(const Factor<__nv_bfloat16>& f, uint32_t t, const uint4& y0, const uint4& y1) {
    uint32_t r[16];
    split::product2n(f.x[0].x, f.nx[0].x, y0.x, r[0], r[8]); split::product2n(f.x[0].y, f.nx[0].y, y0.y, r[1], r[9]);
    split::product2n(f.x[1].x, f.nx[1].x, y1.x, r[2], r[10]); split::product2n(f.x[1].y, f.nx[1].y, y1.y, r[3], r[11]);
    split::product2n(f.x[0].z, f.nx[0].z, y0.z, r[4], r[12]); split::product2n(f.x[0].w, f.nx[0].w, y0.w, r[5], r[13]);
    split::product2n(f.x[1].z, f.nx[1].z, y1.z, r[6], r[14]); split::product2n(f.x[1].w, f.nx[1].w, y1.w, r[7], r[15]);
    tmem_st_16x256b_x4(t, r);
}
__device__ __forceinline__ void store_products(const Factor<NarrowBf16>& f, uint32_t t, const uint2& y0, const uint2& y1) {
    uint32_t r[8];
    split::product2n(f.x[0].x, f.nx[0].x, y0.x, r[0], r[4]); split::product2n(f.x[0].y, f.nx[0].y, y0.y, r[1], r[5]);
    split::product2n(f.x[1].x, f.nx[1].x, y1.x, r[2], r[6]); split::product2n(f.x[1].y, f.nx[1].y, y1.y, r[3], r[7]);
    tmem_st_16x256b_x2(t, r);
}
// fp32: minus the upper part (the tensor core negates it again), then the middle and the lower part.  Three instructions take the
// upper part off a pair of products: x y + r, its distance to r, and what is left of x y, which is never rounded as a whole.
template <bool Wide>
__device__ __forceinline__ void store_products_f32(const Factor<float>& f, uint32_t t, const uint4& y0, const uint4& y1) {
    uint32_t r[8], s[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {                        // first row: channels 0 1, 2 3; second row
        const uint4 &x = f.x[i >> 1], &y = i < 2 ? y0 : y1;
        const float x0 = f4(x, 2 * (i & 1)), x1 = f4(x, 2 * (i & 1) + 1), v0 = f4(y, 2 * (i & 1)), v1 = f4(y, 2 * (i & 1) + 1), round = f.r[i >> 1];
        float p0, p1;
        if constexpr (!Wide) {
            float h0 = round, h1 = round;
            ffma2(h0, h1, x0, x1, v0, v1);
            p0 = round; p1 = round;
            ffma2(p0, p1, h0, h1, -1.f, -1.f);
            r[i] = split::pack_upper(p0, p1);
            ffma2(p0, p1, x0, x1, v0, v1);
        } else {                                         // the upper 8 bits
            p0 = -x0 * v0; p1 = -x1 * v1;
            r[i] = split::pack_upper(p0, p1);
            p0 = -split::rest(p0); p1 = -split::rest(p1);
        }
        r[4 + i] = pack_bf16(p0, p1);
        ffma2(p0, p1, bf16_lo(r[4 + i]), bf16_hi(r[4 + i]), -1.f, -1.f);
        s[i] = pack_bf16(p0, p1);
    }
    tmem_st_16x256b_x2(t, r);
    tmem_st_16x256b_x1(t + 16, s);
}
static __device__ __noinline__ void store_products_wide(uint32_t t, uint4 x0, uint4 x1, uint4 y0, uint4 y1) {
    Factor<float> f;
    f.x[0] = x0; f.x[1] = x1; f.r[0] = f.r[1] = 0.f;
    store_products_f32<true>(f, t, y0, y1);
}
// The products of the three taps of a column.
template <typename T>
__device__ __forceinline__ void store_column(const Factor<T>& f, uint32_t t, const typename Cut<T>::piece (&y)[4]) {
    if constexpr (sizeof(T) == 4) {
        if (f.any_wide) {                                // products from 2^112 on
#pragma unroll 1
            for (int dy = 0; dy < 3; ++dy) store_products_wide(t + dy * Cut<T>::tap_cols, f.x[0], f.x[1], dy == 0 ? y[0] : dy == 1 ? y[1] : y[2], dy == 0 ? y[1] : dy == 1 ? y[2] : y[3]);
        } else {
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) store_products_f32<false>(f, t + dy * Cut<T>::tap_cols, y[dy], y[dy + 1]);
        }
    } else {
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) store_products(f, t + dy * Cut<T>::tap_cols, y[dy], y[dy + 1]);
    }
}

// Descriptor of a contraction image; a (plane, tap) further is contract_step.
__device__ __forceinline__ uint64_t contract_desc(uint32_t img) { return umma_smem_desc(img, 768, 128); }
template <typename T> __host__ __device__ constexpr uint32_t contract_step(int plane, int tap) {
    return (uint32_t)((plane * kK2 + tap) * (Cut<T>::channels / 8) * 48);          // in 16-byte units
}
// The MMAs of one tap (row dy of column dx of a plane), issued by one thread.
template <typename T>
__device__ __forceinline__ void issue_contract(uint32_t tmem, uint32_t p_col, uint64_t b, int plane, int dx, int dy) {
    constexpr uint32_t id16 = umma_idesc_bf16(128, 16), id32 = umma_idesc_bf16(128, 32), id48 = umma_idesc_bf16(128, 48);
    constexpr uint32_t group = 16;                                           // 256 bytes on: the weights' next parts
    const uint32_t l = tmem + kColL<T>;
    const bool fresh = plane == 0 && dy == 0, first = fresh && dx == 0;
    if constexpr (sizeof(T) == 2) {
#pragma unroll
        for (int k = 0; k < Cut<T>::channels / 16; ++k) {
            const uint32_t hi = p_col + 8 * k, lo = p_col + Cut<T>::tap_cols / 2 + 8 * k, r = l + 48;
            const uint64_t bk = b + 96 * k;                                  // 1536 bytes on: the next 16 k
            umma_bf16_ts(l + 16 * dx, hi, bk, id16, fresh && k == 0 ? 0u : 1u);
            umma_bf16_ts(r, hi, bk + group, id16, first && k == 0 ? 0u : 1u);
            umma_bf16_ts(r, hi, bk + 2 * group, id16, 1);
            umma_bf16_ts(r, lo, bk, id16 | kIdescNegateA, 1);
            umma_bf16_ts(r, lo, bk + group, id16 | kIdescNegateA, 1);
        }
    } else {                                                                 // column group i of l: 2^-8i of the first
        const uint32_t hi = p_col, mid = p_col + 8, lo = p_col + 16;
        umma_bf16_ts(l + 16, mid, b, id48, first ? 0u : 1u);
        umma_bf16_ts(l + 32, lo, b, id32, 1);
        if (first) {
            umma_bf16_ts(l, hi, b, id16 | kIdescNegateA, 0);
            umma_bf16_ts(l + 16, hi, b + group, id32 | kIdescNegateA, 1);
        } else {
            umma_bf16_ts(l, hi, b, id48 | kIdescNegateA, 1);
        }
    }
}
// The contraction of the lane's pixel (thread = TMEM lane).
template <typename T>
__device__ __forceinline__ void load_contraction(uint32_t quad, float (&l)[kK2]) {
    float u[32], v[32];
    tmem_ld_32x32b_x32(quad + kColL<T>, u);
    tmem_ld_32x32b_x32(quad + kColL<T> + 32, v);
#pragma unroll
    for (int s = 0; s < kK2; ++s) l[s] = sizeof(T) == 2 ? (u[s] + u[16 + s]) + (v[s] + v[16 + s]) : u[s] + (u[16 + s] + (v[s] + v[16 + s]));
}
// exp2(l scale + bias - their largest) in place of l; returns the sum.  The largest l comes off before the scale is applied, so that
// the slots that matter lose nothing to the rounding of a large logit.
__device__ __forceinline__ float softmax_terms(float (&l)[kK2], float scale, const float* bias) {
    float top = l[0], m = -INFINITY, z = 0.f;
#pragma unroll
    for (int s = 1; s < kK2; ++s) top = fmaxf(top, l[s]);
#pragma unroll
    for (int s = 0; s < kK2; ++s) { l[s] = fmaf(l[s] - top, scale, bias[s]); m = fmaxf(m, l[s]); }
#pragma unroll
    for (int s = 0; s < kK2; ++s) { l[s] = fast_exp2(l[s] - m); z += l[s]; }
    return z;
}

// acc[row][channel of the lane] += D chunk (three taps of a column) at `t` times the halo rows of that column, which are
// loaded while the chunk is on its way.  Tap dy meets halo row `row` + dy, or, in the transposed shift, `row` + 2 - dy.
template <bool Transposed = false>
__device__ __forceinline__ void sum_chunk(__nv_bfloat16, uint32_t t, const unsigned char* plane, int row, int col, int tig, float (&acc)[2][8]) {
    uint32_t d[48];
    tmem_ld3_16x256b_x4_nowait(t, t + 32, t + 64, d);
    uint4 y[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) y[r] = halo_piece<__nv_bfloat16>(plane, row + r, col, tig);
    float f[4][8];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        f[r][0] = bf16_lo(y[r].x); f[r][1] = bf16_hi(y[r].x); f[r][2] = bf16_lo(y[r].y); f[r][3] = bf16_hi(y[r].y);
        f[r][4] = bf16_lo(y[r].z); f[r][5] = bf16_hi(y[r].z); f[r][6] = bf16_lo(y[r].w); f[r][7] = bf16_hi(y[r].w);
    }
    tmem_wait_ld48(d);
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                ffma2(acc[r][2 * j], acc[r][2 * j + 1], __uint_as_float(d[16 * dy + 4 * j + 2 * r]), __uint_as_float(d[16 * dy + 4 * j + 2 * r + 1]),
                      f[r + (Transposed ? 2 - dy : dy)][2 * j], f[r + (Transposed ? 2 - dy : dy)][2 * j + 1]);
}
// planes of 16 channels
template <typename T, bool Transposed>
__device__ __forceinline__ void sum_chunk16(uint32_t t, const unsigned char* plane, int row, int col, int tig, float (&acc)[2][4]) {
    uint32_t d[3][8];
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) tmem_ld_16x256b_x2_nowait(t + 16 * dy, d[dy]);
    float f[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const typename Cut<T>::piece y = halo_piece<T>(plane, row + r, col, tig);
        if constexpr (sizeof(T) == 2) { f[r][0] = bf16_lo(y.x); f[r][1] = bf16_hi(y.x); f[r][2] = bf16_lo(y.y); f[r][3] = bf16_hi(y.y); }
        else { f[r][0] = f4(y, 0); f[r][1] = f4(y, 1); f[r][2] = f4(y, 2); f[r][3] = f4(y, 3); }
    }
    tmem_wait_ld();
#pragma unroll
    for (int dy = 0; dy < 3; ++dy) {
        tmem_pass(d[dy]);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                ffma2(acc[r][2 * j], acc[r][2 * j + 1], __uint_as_float(d[dy][4 * j + 2 * r]), __uint_as_float(d[dy][4 * j + 2 * r + 1]),
                      f[r + (Transposed ? 2 - dy : dy)][2 * j], f[r + (Transposed ? 2 - dy : dy)][2 * j + 1]);
    }
}
template <bool Transposed = false>
__device__ __forceinline__ void sum_chunk(float, uint32_t t, const unsigned char* plane, int row, int col, int tig, float (&acc)[2][4]) {
    sum_chunk16<float, Transposed>(t, plane, row, col, tig, acc);
}
template <bool Transposed = false>
__device__ __forceinline__ void sum_chunk(NarrowBf16, uint32_t t, const unsigned char* plane, int row, int col, int tig, float (&acc)[2][4]) {
    sum_chunk16<NarrowBf16, Transposed>(t, plane, row, col, tig, acc);
}

}  // namespace team
}  // namespace slide_attn
