// Quantisation step of the alternating refinement (Alg. 1, step 2.1; Sec. 3.3): with B and A fixed,
//
//     Q_ij = argmin over the codes c of (S_ij * L[c] - W_ij)^2,      S = B A (Eq. 3),
//
// written out as packed codes in the library's layout.  The paper does not say which level wins a tie:
// the lowest code does.  S is rebuilt tile by tile on the tensor cores exactly as the forward kernels
// rebuild it (bf16 operands from shared memory, fp32 in TMEM, never stored in full).  The decision is
// taken in fp32 with S accumulated in fp32, in one of three ways (chosen on the host from the level table):
//   buckets   ascending table whose midpoints lie further apart than a bucket is wide (every NormalFloat table): the
//             approximate ratio W / S picks a bucket, the bucket gives the one midpoint in it and the code below,
//             and one exact comparison decides (about thirteen instructions a weight);
//   bisection any other ascending table: log2 of the level count products and comparisons per weight;
//   trial     any other table: every level in turn (one fused multiply-add and a square per level).
//
// A step is a tile of 128 rows and 64 columns.  One CTA per SM takes an equal run of the steps of the whole weight, row tile after row
// tile (two CTAs per SM, or several rounds of CTAs, paid the set-up of a CTA, worth about three steps, once more: 4096 x 4096 33 us
// against 20).  Warp roles (18 warps):
//   0..15 search, two groups of eight on alternating steps (three groups have to make do with 72 registers: 14336 x 4096, 4 bits, 55 us
//         against 49): a thread owns one row and 32 of the step's columns, 16 at a time: its S from TMEM, its weights from the W
//         tile in shared memory (TMA, 128-byte swizzle: row-wise reads from global memory would touch 32 lines each).
//   16    TMEM allocation and MMA issuer: S[128 x 64] = B_tile (128 x r) * A_tile (r x 64) into one of
//         four TMEM buffers, as soon as the factor tile has landed and the buffer has been read.
//   17    TMA producer of the W tiles, the factor tiles A[:, step] and, where a row tile begins, B_tile.
// Every wait is bounded; on expiry the role records LORDS_ERR_TIMEOUT and leaves its loop.
//
// Bound: instructions per weight (about 20 with packing) and the latency of their chain.  14336 x 4096, 3 bits, r = 48: 90 us with
// bisection and weights read row by row from global memory, 51 now; 4096 x 4096, 4 bits, r = 32: 47 -> 20; r = 128, on the CUDA
// cores before: 834 -> 60.
//
// Rows of W or A that are not 16-byte multiples (n not a multiple of 8) are copied to padded rows in the workspace first; without
// room there, and for small layers off the tile grid, a plain CUDA-core kernel runs.
//
// Layers with a ragged row (n not a multiple of 64) or a rank above 64 ran on the CUDA cores before, whose sums (rounded to nearest) and
// comparison of errors (one rounding of a small difference) are nearer to the exact decision than the tensor cores' S, which is cut off,
// and a rounded product.  For them (SURE) a weight that lies nearer to a midpoint than S and the midpoint may be off is decided in
// 64 bits: their codes are the exact ones (of 1.2e9 weights none differs from the decision in 64 bits; on the CUDA cores 1 to 7 of 16.8 M at
// r = 128 did).  4096 x 4096, r = 128: 60 us a call, 180 with factors of mixed sign, whose S cancels (CUDA cores 834; 19 with the tensor cores'
// S for every decision); 5472 x 10524, r = 6: 227 (437; 199).
#include <cuda.h>
#include <cuda_bf16.h>

#include "lords_internal.h"
#include "lords_ptx.cuh"
#include "lords_tc_common.cuh"

namespace lords {

namespace {

using namespace ptx;

constexpr int kRowsQ = 128;                    // rows of W per CTA = UMMA M
constexpr int kColsQ = 64;                     // columns per step
constexpr int kSearchWarps = 8;                // warps of a step
constexpr int kGroupsQ = 2;                    // groups of search warps, on alternating steps
constexpr int kIssuerWarpQ = kGroupsQ * kSearchWarps;     // 16
constexpr int kTmaWarpQ = kIssuerWarpQ + 1;               // 17
constexpr int kThreadsQ = (kTmaWarpQ + 1) * 32;
constexpr int kSAQ = 4;                        // factor-tile ring depth
constexpr int kSWQ = 6;                        // weight-tile ring depth
constexpr int kSDQ = 4;                        // S buffers in TMEM
static_assert(kSWQ % kGroupsQ == 0 && kSDQ % kGroupsQ == 0, "a buffer is always read by the same group");
constexpr uint32_t kTmemColsQ = kSDQ * kColsQ;
constexpr int kWTileQ = kRowsQ * 128;          // 128 rows x 64 columns bf16

enum Search { kBuckets, kBisect, kTrial };

// BITS: code width.  RA: ranks the factor tiles are sized for (64 or 128).
template <int BITS, int RA> struct QuantCfg {
    static constexpr int BUCKETS = BITS == 4 ? 64 : BITS == 3 ? 32 : 16;
    static constexpr int LUT = BUCKETS * 256;                 // 32 lane-private copies of {midpoint, code below}
    static constexpr int ATILE = RA * 128;
    static constexpr int BTILE = RA / 64 * kRowsQ * 128;
    static constexpr int STAGE = BITS == 4 ? 0 : 32 * BITS * 4;       // packed codes of a warp's 32 rows (see store_codes_staged)
    static constexpr int SMEM = 1024 + kSWQ * kWTileQ + kSAQ * ATILE + BTILE + LUT + 256 + kGroupsQ * kSearchWarps * STAGE;
};

struct alignas(64) QuantParams {
    CUtensorMap tm_a;     // bf16 [r][n], box {64, r_pad}, 128-byte swizzle (ranks past r and columns past n read as zero)
    CUtensorMap tm_w;     // bf16 [m][n], box {64, 128}, 128-byte swizzle (rows past m and columns past n read as zero)
    CUtensorMap tm_b;     // bf16 [m][r], box {64, 128}, 128-byte swizzle; used if rows of B are 16-byte multiples
    const uint16_t *B;    // bf16 [m][r]
    const uint16_t *A;    // bf16 [r][n]
    const float *a_norm;  // SURE: per step, how far S of a row of norm 1 may put a weight from its midpoint
    const float *b_norm;  // SURE: per row, the norm of its B
    uint8_t *Q;           // packed codes, row pitch n * bits / 8
    float levels[16];
    float mids[16];       // ascending table: mids[c] = (levels[c] + levels[c + 1]) / 2
    float bucket_mid[64]; // the midpoint in (or next to) bucket k, +infinity if there is none above its lower edge
    uint8_t bucket_code[64];   // midpoints below it
    float least_scale;    // SURE: |S| has to be more than this times what it may be off for the bucket to be the right one
    float bucket_scale, bucket_bias;   // bucket of a ratio t: saturate(t * scale + bias) * (buckets - 1), rounded
    int m, n, r, r_pad;
    int steps;            // 64-column steps per row tile
    int row_splits;       // 0: all steps of all row tiles in equal runs; else ranges per row tile (a run stays in its row tile)
    int row_tiles;
    int *status;
};

// The code whose level is nearest to w / s: every level in turn, the first (lowest) code keeps a tie.
template <int LEVELS>
__device__ __forceinline__ uint32_t nearest_code(float s, float w, const float (&lv)[16])
{
    uint32_t best = 0;
    const float d0 = fmaf(s, lv[0], -w);
    float e_best = d0 * d0;
#pragma unroll
    for (int c = 1; c < LEVELS; ++c) {
        const float d = fmaf(s, lv[c], -w);
        const float e = d * d;
        if (e < e_best) { e_best = e; best = (uint32_t)c; }
    }
    return best;
}

// The same for a strictly ascending table, by bisection over the midpoints between neighbouring levels:
// (s v - w)^2 = s^2 (v - w/s)^2, so the nearest level to t = w / s wins whatever the sign of s, and
// t > mid  <=>  b > a mid  with a = |s|, b = w sign(s).  The code is the number of midpoints below t; a
// weight exactly on a midpoint keeps the lower code, and s = 0 (every level equally good) gives code 0.
// The thresholds of the later steps are picked by selects on the earlier outcomes: log2(LEVELS)
// products and comparisons instead of LEVELS.
template <int LEVELS>
__device__ __forceinline__ uint32_t nearest_code_sorted(float s, float w, const float (&md)[16])
{
    const float a = fabsf(s);
    float b = s < 0.0f ? -w : w;
    b = a == 0.0f ? -INFINITY : b;
    if constexpr (LEVELS == 16) {
        const bool p3 = b > a * md[7];
        const bool p2 = b > a * (p3 ? md[11] : md[3]);
        const float m1 = p3 ? (p2 ? md[13] : md[9]) : (p2 ? md[5] : md[1]);
        const bool p1 = b > a * m1;
        const float m0hi = p2 ? (p1 ? md[14] : md[12]) : (p1 ? md[10] : md[8]);
        const float m0lo = p2 ? (p1 ? md[6] : md[4]) : (p1 ? md[2] : md[0]);
        const bool p0 = b > a * (p3 ? m0hi : m0lo);
        return ((uint32_t)p3 << 3) | ((uint32_t)p2 << 2) | ((uint32_t)p1 << 1) | (uint32_t)p0;
    } else if constexpr (LEVELS == 8) {
        const bool p2 = b > a * md[3];
        const bool p1 = b > a * (p2 ? md[5] : md[1]);
        const float m0 = p2 ? (p1 ? md[6] : md[4]) : (p1 ? md[2] : md[0]);
        const bool p0 = b > a * m0;
        return ((uint32_t)p2 << 2) | ((uint32_t)p1 << 1) | (uint32_t)p0;
    } else {
        const bool p1 = b > a * md[1];
        const bool p0 = b > a * (p1 ? md[2] : md[0]);
        return ((uint32_t)p1 << 1) | (uint32_t)p0;
    }
}

// The exact decision: S in 64 bits (products of bf16 are exact there), every level in turn.
template <int LEVELS>
__device__ __noinline__ uint32_t exact_code(const QuantParams &p, int i, int j, float w)
{
    const uint16_t *b = p.B + (size_t)i * p.r, *a = p.A + j;
    double s = 0.0;
    for (int k = 0; k < p.r; ++k)         // (unrolled sixteen times it is slower: r = 128, mixed signs, 409 us against 260)
        s = fma((double)__uint_as_float((uint32_t)b[k] << 16), (double)__uint_as_float((uint32_t)a[(size_t)k * p.n] << 16), s);
    uint32_t best = 0;
    double e_best = 0.0;
    for (int c = 0; c < LEVELS; ++c) {
        const double d = fma(s, (double)p.levels[c], -(double)w), e = d * d;
        if (c == 0 || e < e_best) { e_best = e; best = (uint32_t)c; }
    }
    return best;
}
// Code c of the 32 in `packed` replaced.
template <int BITS> __device__ __forceinline__ void replace_code(uint32_t (&packed)[BITS], int c, uint32_t code)
{
    constexpr uint32_t mask = (1u << BITS) - 1u;
    const int at = c * BITS >> 5, sh = c * BITS & 31;
#pragma unroll
    for (int k = 0; k < BITS; ++k) {
        if (k == at) packed[k] = (packed[k] & ~(mask << sh)) | code << sh;
        if (k == at + 1 && sh + BITS > 32) packed[k] = (packed[k] & ~(mask >> (32 - sh))) | code >> (32 - sh);
    }
}

// The first `count` of 32 codes of one row -> packed bytes at `dst` (the row's byte offset of these 32 columns); w: the codes packed, BITS
// words.  `words`: dst is 4-byte aligned; 16-byte aligned rows of 4-bit codes go out as one word.
template <int BITS> __device__ __forceinline__ void store_codes(uint8_t *dst, const uint32_t (&w)[BITS], int count, bool words, bool vec)
{
    if (count >= 32 && words) {
        if (BITS == 4 && vec) {
            *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[BITS > 2 ? 2 : 0], w[BITS > 3 ? 3 : 0]);
        } else {
#pragma unroll
            for (int k = 0; k < BITS; ++k) reinterpret_cast<uint32_t *>(dst)[k] = w[k];
        }
    } else if (count >= 32) {
        store_words_anywhere<BITS>(dst, w);
    } else {
#pragma unroll
        for (int k = 0; k < 4 * BITS; ++k)
            if (8 * k < count * BITS) dst[k] = (uint8_t)(w[k >> 2] >> (8 * (k & 3)));
    }
}

// EDGE: some tile reaches past the matrix (a variant of its own: the check costs the others 3 %).  SURE: close decisions in 64 bits.
template <int BITS, int MODE, int RA, bool EDGE, bool SURE>
__global__ void __launch_bounds__(kThreadsQ, 1) lords_quantize_kernel(const __grid_constant__ QuantParams p)
{
    using C = QuantCfg<BITS, RA>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t w0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a0 = w0 + kSWQ * kWTileQ, b_tile = a0 + kSAQ * C::ATILE, lut = b_tile + C::BTILE, bars = lut + C::LUT;
    const uint32_t bar_w = bars, bar_w_free = bar_w + 8 * kSWQ, bar_a = bar_w_free + 8 * kSWQ, bar_a_free = bar_a + 8 * kSAQ;
    const uint32_t bar_s = bar_a_free + 8 * kSAQ, bar_s_free = bar_s + 8 * kSDQ, bar_b = bar_s_free + 8 * kSDQ, tmem_slot = bar_b + 8;
    static_assert(16 * (kSWQ + kSAQ + kSDQ) + 8 + 4 <= 256, "barrier area");
    // SURE: with tries one after the other 3 bits take 24 to 31 % longer (2216 x 12576, rank 65: 59 us, 74 so; rank 100: 70 and 92; 2 and 4 bits are
    // level).  The other forms, alone, are within 1 % either way; a training step of 4096 x 4096 at 1024 tokens takes 205.5 us so, 207.2 with sleeps.
    constexpr int kSleep = SURE ? kWaitSleepNs : 0;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // this CTA's run of steps, across row tiles (step `st` of row tile `rt` is number rt * steps + st)
    int rt0, st0, total;
    if (p.row_splits == 0) {
        const long long all = (long long)p.row_tiles * p.steps;
        const long long g0 = all * blockIdx.x / gridDim.x, g1 = all * (blockIdx.x + 1) / gridDim.x;
        rt0 = (int)(g0 / p.steps);
        st0 = (int)(g0 % p.steps);
        total = (int)(g1 - g0);
    } else {
        const int s = (int)blockIdx.x % p.row_splits;
        rt0 = (int)blockIdx.x / p.row_splits;
        st0 = (int)((long long)p.steps * s / p.row_splits);
        total = (int)((long long)p.steps * (s + 1) / p.row_splits) - st0;
    }
    const bool b_by_tma = (p.r & 7) == 0;
    const int *status = p.status;
    bool failed = false;

    if (warp == kTmaWarpQ) {
        if (lane == 0) {
            for (int b = 0; b < kSWQ; ++b) { mbar_init(bar_w + 8 * b, 1); mbar_init(bar_w_free + 8 * b, kSearchWarps); }
            for (int b = 0; b < kSAQ; ++b) { mbar_init(bar_a + 8 * b, 1); mbar_init(bar_a_free + 8 * b, 1); }
            for (int b = 0; b < kSDQ; ++b) { mbar_init(bar_s + 8 * b, 1); mbar_init(bar_s_free + 8 * b, kSearchWarps); }
            mbar_init(bar_b, 1);
            fence_mbar_init();
            tma_prefetch_desc(&p.tm_w);
            tma_prefetch_desc(&p.tm_a);
        }
    } else if (warp == kIssuerWarpQ) {
        tmem_alloc(tmem_slot, kTmemColsQ);
        tmem_relinquish();
    } else {
        if (MODE == kBuckets)
            for (int k = warp; k < C::BUCKETS; k += kIssuerWarpQ)
                asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(lut + (uint32_t)(k * 256 + lane * 8)), "r"(__float_as_uint(p.bucket_mid[k])),
                             "r"((uint32_t)p.bucket_code[k]) : "memory");
        if (!b_by_tma && warp < kSearchWarps) {
            // rows of B that are not 16-byte multiples: element by element, zeros past rank r and past row m
            const int rr = tid >> 1, i = rt0 * kRowsQ + rr;
            for (int c = 0; c < RA / 16; ++c) {
                const int chunk = (tid & 1) * (RA / 16) + c;
                uint32_t w4[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int k = chunk * 8 + e * 2;
                    const uint32_t lo = (i < p.m && k < p.r) ? p.B[(size_t)i * p.r + k] : 0u;
                    const uint32_t hi = (i < p.m && k + 1 < p.r) ? p.B[(size_t)i * p.r + k + 1] : 0u;
                    w4[e] = lo | (hi << 16);
                }
                sts_v4(b_tile + (uint32_t)((chunk >> 3) * kRowsQ * 128 + (rr >> 3) * 1024 + (rr & 7) * 128 + (((chunk & 7) ^ (rr & 7)) * 16)),
                       make_uint4(w4[0], w4[1], w4[2], w4[3]));
            }
            fence_proxy_async_smem();
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));

    if (warp == kTmaWarpQ) {
        if (lane == 0) {
            int next_w = 0, w_rt = rt0, w_st = st0;          // weight tiles run ahead of the factor tiles as far as their ring allows
            int rt = rt0, st = st0;
            for (int it = 0; it < total; ++it) {
                if (b_by_tma && (it == 0 || st == 0)) {      // a new row tile: its B once nothing reads the last one's
                    if (it > 0 && !mbar_wait<kSleep>(bar_a_free + 8 * ((it - 1) % kSAQ), (uint32_t)(((it - 1) / kSAQ) & 1), status, 29)) { failed = true; break; }
                    mbar_expect_tx(bar_b, (uint32_t)C::BTILE);
                    for (int h = 0; h < RA / 64; ++h) tma_load_2d(b_tile + (uint32_t)(h * kRowsQ * 128), &p.tm_b, h * 64, rt * kRowsQ, bar_b);
                }
                while (next_w < total && next_w < it + kSWQ) {
                    const int s = next_w % kSWQ;
                    if (next_w >= kSWQ) {
                        const uint32_t par = (uint32_t)((next_w / kSWQ - 1) & 1);
                        if (next_w > it) { if (!mbar_try_wait(bar_w_free + 8 * s, par)) break; }
                        else if (!mbar_wait<kSleep>(bar_w_free + 8 * s, par, status, 30)) { failed = true; break; }
                    }
                    mbar_expect_tx(bar_w + 8 * s, (uint32_t)kWTileQ);
                    tma_load_2d(w0 + (uint32_t)(s * kWTileQ), &p.tm_w, w_st * kColsQ, w_rt * kRowsQ, bar_w + 8 * s);
                    ++next_w;
                    if (++w_st == p.steps) { w_st = 0; ++w_rt; }
                }
                if (failed) break;
                const int sa = it % kSAQ;
                if (it >= kSAQ && !mbar_wait<kSleep>(bar_a_free + 8 * sa, (uint32_t)((it / kSAQ - 1) & 1), status, 31)) { failed = true; break; }
                mbar_expect_tx(bar_a + 8 * sa, (uint32_t)(p.r_pad * 128));
                tma_load_2d(a0 + (uint32_t)(sa * C::ATILE), &p.tm_a, st * kColsQ, 0, bar_a + 8 * sa);
                if (++st == p.steps) { st = 0; ++rt; }
            }
        }
        __syncwarp();
    } else if (warp == kIssuerWarpQ) {
        const uint32_t tmem_u = warp_uniform(tmem_base), leader = elect_one();
        constexpr uint32_t idesc = umma_idesc_f16(1, 0, 1, kRowsQ, kColsQ);     // bf16, B operand MN-major, N = 64
        const uint32_t desc_hi = (uint32_t)(umma_desc_sw128(0, 1024, 16) >> 32);
        const uint32_t lbo_lo = (uint32_t)umma_desc_sw128(0, 1024, 16);
        const uint32_t b_lo = lbo_lo | ((b_tile & 0x3FFFFu) >> 4), a_lo0 = lbo_lo | ((a0 & 0x3FFFFu) >> 4);
        uint32_t b_phase = 0;
        int st = st0;
        for (int it = 0; it < total; ++it) {
            if (b_by_tma && (it == 0 || st == 0)) {
                if (!mbar_wait_warp<kSleep>(bar_b, b_phase, status, 36)) { failed = true; break; }
                b_phase ^= 1;
            }
            if (++st == p.steps) st = 0;
            const int sa = it % kSAQ, sd = it % kSDQ;
            if (!mbar_wait_warp2<kSleep>(bar_a + 8 * sa, (uint32_t)((it / kSAQ) & 1), bar_s_free + 8 * sd, (uint32_t)((it / kSDQ + 1) & 1), status, 32)) { failed = true; break; }
            tc_fence_after_sync();
            const uint32_t a_lo = a_lo0 + (uint32_t)(sa * (C::ATILE >> 4));
            for (int k = 0; k < p.r_pad / 16; ++k)
                umma_f16_ss(tmem_u + (uint32_t)(sd * kColsQ), umma_desc_pack(b_lo + (k >> 2) * (kRowsQ * 128 >> 4) + (k & 3) * 2, desc_hi),
                            umma_desc_pack(a_lo + k * 128, desc_hi), idesc, k > 0, leader);
            umma_commit(bar_s + 8 * sd, leader);
            umma_commit(bar_a_free + 8 * sa, leader);
        }
        // no commit is still on its way to a barrier when the CTA ends
        if (!failed && total > 0 && !mbar_wait_warp<kSleep>(bar_a_free + 8 * ((total - 1) % kSAQ), (uint32_t)(((total - 1) / kSAQ) & 1), status, 34)) failed = true;
    } else {
        const int q = warp & 3, ch = (warp >> 2) & 1, row = q * 32 + lane;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * 32);
        const uint32_t w_row = w0 + (uint32_t)((row >> 3) * 1024 + (row & 7) * 128), lut_lane = lut + 8u * (uint32_t)lane;
        // the bucket's number arrives as the low bits of a float of magnitude 2^23: its bits times 256, less what the exponent adds
        const uint32_t lut_magic = lut_lane - 0x4B000000u * 256u;
        float lv[MODE == kBuckets ? 1 : 16];
        if constexpr (MODE != kBuckets) {
#pragma unroll
            for (int c = 0; c < 16; ++c) lv[c] = MODE == kBisect ? p.mids[c] : p.levels[c];
        }
        const size_t qpitch = (size_t)p.n * BITS / 8;
        const bool words = (qpitch & 3) == 0, vec = (qpitch & 15) == 0;
        const int group = warp / kSearchWarps;
        const uint32_t stage = bars + 256u + (uint32_t)(warp * C::STAGE);
        int rt = rt0, st = st0 + group, b_row = -1;
        float b_norm = 0.0f;
        for (int it = group; it < total; it += kGroupsQ) {
            while (st >= p.steps) { st -= p.steps; ++rt; }
            const int sd = it % kSDQ, sw = it % kSWQ, col0 = st * kColsQ + ch * 32, i = rt * kRowsQ + row;
            float off = 0.0f, least_s = 0.0f;                // SURE: a product of S and a midpoint is off by no more than this
            if constexpr (SURE) {
                if (i != b_row) { b_row = i; b_norm = i < p.m ? __ldg(p.b_norm + i) : 0.0f; }
                off = b_norm * __ldg(p.a_norm + st);
                least_s = off * p.least_scale;
            }
            st += kGroupsQ;
            if (!mbar_wait_warp2<kSleep>(bar_s + 8 * sd, (uint32_t)((it / kSDQ) & 1), bar_w + 8 * sw, (uint32_t)((it / kSWQ) & 1), status, 35)) { failed = true; break; }
            tc_fence_after_sync();
            const float past = EDGE && (i >= p.m || col0 >= p.n) ? 1.0f : 0.0f;
            uint32_t packed[BITS];
#pragma unroll
            for (int k = 0; k < BITS; ++k) packed[k] = 0u;
#pragma unroll
            for (int h = 0; h < 2; ++h) {                    // 16 columns at a time: all of the weights at once would not fit the registers
                uint32_t s[16];
                tmem_ld_32x16(lane_addr + (uint32_t)(sd * kColsQ + h * 16), s);
                const uint32_t at = w_row + (uint32_t)(sw * kWTileQ);
                uint32_t unsure = 0;                         // SURE: a bit per column
                const uint4 wv[2] = {lds_v4(at + (uint32_t)(((ch * 4 + h * 2) ^ (row & 7)) << 4)), lds_v4(at + (uint32_t)(((ch * 4 + h * 2 + 1) ^ (row & 7)) << 4))};
                tmem_wait_ld(s);
                if (h == 1) {
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_s_free + 8 * sd);      // S is in registers: the buffer may be refilled
                }
                auto weight = [&](int c) {
                    const uint4 &v = wv[(c >> 3) & 1];
                    const uint32_t u = (c & 7) / 2 == 0 ? v.x : (c & 7) / 2 == 1 ? v.y : (c & 7) / 2 == 2 ? v.z : v.w;
                    return __uint_as_float((c & 1) ? (u & 0xFFFF0000u) : (u << 16));
                };
                auto pack = [&](auto code_of) {
#pragma unroll
                    for (int c = h * 16; c < h * 16 + 16; ++c) {
                        const uint32_t code = code_of(c);
                        const int bit = c * BITS, wi = bit >> 5, sh = bit & 31;
                        packed[wi] += code << sh;
                        if (sh + BITS > 32) packed[wi + 1 < BITS ? wi + 1 : wi] += code >> (32 - sh);
                    }
                };
                if constexpr (MODE == kBuckets) {
                    // a scale outside (2^-100, 2^100) (zero above all: code 0) takes the exact products, and so does the warp with it; rows and
                    // columns past the matrix have scale zero and are not stored, so they have no say (6001 x 2048: the warps of the
                    // last row tile were the whole call's tail, 35 us against 16)
                    float least = fabsf(__uint_as_float(s[0])), most = least;
#pragma unroll
                    for (int c = 1; c < 16; ++c) {
                        least = fminf(least, fabsf(__uint_as_float(s[c])));
                        most = fmaxf(most, fabsf(__uint_as_float(s[c])));
                    }
                    if (__all_sync(0xffffffffu, (EDGE ? fmaxf(least, past) : least) > 7.8886e-31f && most < 1.2676e30f)) {
                        const uint64_t top2 = f32x2((float)(C::BUCKETS - 1), (float)(C::BUCKETS - 1)), magic2 = f32x2(8388608.0f, 8388608.0f);
                        float f[2];
                        pack([&](int c) {
                            const float w = weight(c);
                            if ((c & 1) == 0) {
                                // two buckets at a time: round(saturate(t * scale + bias) * (buckets - 1)) as the low bits of a float
                                float t[2];
                                f32x2_split(f32x2_mul(f32x2(w, weight(c + 1)), f32x2(rcp_approx(__uint_as_float(s[c & 15])), rcp_approx(__uint_as_float(s[(c + 1) & 15])))), t[0], t[1]);
                                const float u = __saturatef(fmaf(t[0], p.bucket_scale, p.bucket_bias)), v = __saturatef(fmaf(t[1], p.bucket_scale, p.bucket_bias));
                                f32x2_split(f32x2_fma(f32x2(u, v), top2, magic2), f[0], f[1]);
                            }
                            uint32_t mid, below, above;
                            asm("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(mid), "=r"(below) : "r"(__float_as_uint(f[c & 1]) * 256u + lut_magic));
                            // t > mid  <=>  w sign(s) > |s| mid (as in the bisection)
                            const float b = __uint_as_float(__float_as_uint(w) ^ (s[c & 15] & 0x80000000u));
                            if constexpr (SURE) {
                                const float d = fmaf(-fabsf(__uint_as_float(s[c & 15])), __uint_as_float(mid), b);
                                asm("set.gt.u32.f32 %0, %1, %2;" : "=r"(above) : "f"(d), "f"(0.0f));
                                if (!(fabsf(d) > off && fabsf(__uint_as_float(s[c & 15])) > least_s && fabsf(w) < INFINITY)) unsure |= 1u << (c & 15);
                                return below - above;
                            }
                            asm("set.gt.u32.f32 %0, %1, %2;" : "=r"(above) : "f"(b), "f"(fabsf(__uint_as_float(s[c & 15])) * __uint_as_float(mid)));
                            return below - above;             // the outcome is 0 or -1
                        });
                    } else if constexpr (SURE) {
                        pack([](int) { return 0u; });
                        unsure = 0xFFFFu;
                    } else {
                        // the bisection's answer by counting, which needs no registers for its thresholds
                        pack([&](int c) {
                            const float sc = __uint_as_float(s[c & 15]), a = fabsf(sc), w = weight(c), b = a == 0.0f ? -INFINITY : sc < 0.0f ? -w : w;
                            uint32_t code = 0;
#pragma unroll
                            for (int l = 0; l + 1 < (1 << BITS); ++l) code += b > a * p.mids[l] ? 1u : 0u;
                            return code;
                        });
                    }
                    if constexpr (SURE) {
                        const int left = i < p.m ? p.n - col0 - h * 16 : 0;          // columns of the sixteen that exist
                        unsure &= left >= 16 ? 0xFFFFu : left > 0 ? (1u << left) - 1u : 0u;
                        if (__any_sync(0xffffffffu, unsure != 0u)) {
                            for (; unsure != 0u; unsure &= unsure - 1u) {
                                const int c = h * 16 + __ffs((int)unsure) - 1;
                                float w = 0.0f;
#pragma unroll
                                for (int e = h * 16; e < h * 16 + 16; ++e) w = e == c ? weight(e) : w;
                                replace_code<BITS>(packed, c, exact_code<(1 << BITS)>(p, i, col0 + c, w));
                            }
                            __syncwarp();
                        }
                    }
                } else if constexpr (MODE == kBisect) {
                    pack([&](int c) { return nearest_code_sorted<(1 << BITS)>(__uint_as_float(s[c & 15]), weight(c), lv); });
                } else {
                    pack([&](int c) { return nearest_code<(1 << BITS)>(__uint_as_float(s[c & 15]), weight(c), lv); });
                }
            }
            if (BITS != 4 && words && p.n - col0 >= 32)
                store_codes_staged<BITS>(stage, p.Q + (size_t)(rt * kRowsQ + q * 32) * qpitch + (size_t)col0 * BITS / 8, qpitch, p.m - rt * kRowsQ - q * 32, lane, packed);
            else if (i < p.m && col0 < p.n) store_codes<BITS>(p.Q + (size_t)i * qpitch + (size_t)col0 * BITS / 8, packed, p.n - col0, words, vec);
            // only now that the weights have been used: an arrival can overtake loads that are still in flight
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_w_free + 8 * sw);
        }
    }

    if (failed) ptx::record_give_up(p.status, LORDS_ERR_TIMEOUT);
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kIssuerWarpQ) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemColsQ);
    }
}

// Plain CUDA-core version for any shape: a thread owns one row and one pack group of 32 columns (or what
// is left of the row), S by a loop over the ranks in fp32, the same level search.
template <int BITS>
__global__ void lords_quantize_simt_kernel(const uint16_t *__restrict__ W, const uint16_t *__restrict__ B,
                                           const uint16_t *__restrict__ A, uint8_t *__restrict__ Q, int m, int n, int r,
                                           const float *__restrict__ levels_dev)
{
    constexpr int LEVELS = 1 << BITS;
    constexpr int G = BITS == 3 ? 32 : (BITS == 4 ? 2 : 4);        // codes per whole number of bytes
    float lv[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) lv[c] = c < LEVELS ? levels_dev[c] : 0.0f;
    const long long groups_per_row = n / G;
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long long)m * groups_per_row) return;
    const int i = (int)(gid / groups_per_row);
    const int j0 = (int)(gid % groups_per_row) * G;
    unsigned long long lo = 0;
    uint32_t hi = 0;
    for (int g = 0; g < G; ++g) {
        const int j = j0 + g;
        float s = 0.0f;
        for (int k = 0; k < r; ++k)
            s = fmaf(__uint_as_float((uint32_t)B[(size_t)i * r + k] << 16), __uint_as_float((uint32_t)A[(size_t)k * n + j] << 16), s);
        const uint32_t c = nearest_code<LEVELS>(s, __uint_as_float((uint32_t)W[(size_t)i * n + j] << 16), lv);
        const int bit = g * BITS;
        if (bit < 64) lo |= (unsigned long long)c << bit;
        if (bit + BITS > 64) hi |= bit >= 64 ? c << (bit - 64) : c >> (64 - bit);
    }
    uint8_t *dst = Q + (size_t)i * ((size_t)n * BITS / 8) + (size_t)j0 * BITS / 8;
    constexpr int BYTES = G * BITS / 8;
#pragma unroll
    for (int b = 0; b < BYTES; ++b) dst[b] = b < 8 ? (uint8_t)(lo >> (8 * b)) : (uint8_t)(hi >> (8 * (b - 8)));
}

// Blocks below `steps`: how far S of a row of norm 1 may put a weight from a midpoint, over the 64 columns of a step, i.e. `scale` times the
// largest norm of a column of A.  The others: norms of eight rows of B each.
__global__ void __launch_bounds__(256) lords_quantize_norms_kernel(const uint16_t *__restrict__ B, const uint16_t *__restrict__ A, int m, int n, int r,
                                                                   int steps, float scale, float *__restrict__ a_norm, float *__restrict__ b_norm)
{
    __shared__ float part[256];                     // (squares in 64 bits: those of factors below 1e-19 or above 1e19 leave the range of a float)
    const int tid = threadIdx.x, lane = tid & 31;
    double sum = 0.0;
    if ((int)blockIdx.x < steps) {
        const int j = (int)blockIdx.x * kColsQ + (tid & 63);
        if (j < n)
            for (int k = tid >> 6; k < r; k += 4) {
                const double v = __uint_as_float((uint32_t)A[(size_t)k * n + j] << 16);
                sum = fma(v, v, sum);
            }
        part[tid] = (float)sqrt(sum);
        __syncthreads();
        if (tid < 32) {
            float most = 0.0f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                double four = 0.0;
#pragma unroll
                for (int q = 0; q < 4; ++q) four = fma((double)part[tid + 32 * h + 64 * q], (double)part[tid + 32 * h + 64 * q], four);
                most = fmaxf(most, (float)sqrt(four));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, o));
            if (tid == 0) a_norm[blockIdx.x] = scale * most;
        }
    } else {
        const int i = ((int)blockIdx.x - steps) * 8 + (tid >> 5);
        if (i >= m) return;
        for (int k = lane; k < r; k += 32) {
            const double v = __uint_as_float((uint32_t)B[(size_t)i * r + k] << 16);
            sum = fma(v, v, sum);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) b_norm[i] = (float)sqrt(sum);
    }
}

template <int BITS, int MODE, int RA, bool EDGE, bool SURE> int launch_quantize_tc(QuantParams &k, const State &st, cudaStream_t stream)
{
    static bool done[kMaxDevices] = {};
    const int dev = device_slot(st);
    if (!done[dev]) {
        LORDS_CUDA_TRY(cudaFuncSetAttribute(lords_quantize_kernel<BITS, MODE, RA, EDGE, SURE>, cudaFuncAttributeMaxDynamicSharedMemorySize, QuantCfg<BITS, RA>::SMEM));
        done[dev] = true;
    }
    // One run of steps per CTA that can be resident: setting a CTA up costs as much as about three steps, which a second round of CTAs
    // would pay again, and equal runs leave no partial round.  With the B tile built element by element (rank not a multiple of 8)
    // a run stays within its row tile: the least rounds times (steps + 3) then.
    k.row_tiles = (k.m + kRowsQ - 1) / kRowsQ;
    const long long all = (long long)k.row_tiles * k.steps, resident = st.sm_count;
    long long grid = all < resident ? all : resident;
    k.row_splits = 0;
    if ((k.r & 7) != 0) {
        double best = 1e30;
        for (int s = 1; s <= k.steps && s <= 4096; ++s) {
            const double t = (double)(((long long)k.row_tiles * s + resident - 1) / resident) * ((k.steps + s - 1) / s + 3.0);
            if (t < best) { best = t; k.row_splits = s; }
        }
        grid = (long long)k.row_tiles * k.row_splits;
    }
    if (grid > 2147483647LL) return LORDS_ERR_SHAPE;
    lords_quantize_kernel<BITS, MODE, RA, EDGE, SURE><<<(unsigned)grid, kThreadsQ, QuantCfg<BITS, RA>::SMEM, stream>>>(k);
    LORDS_CUDA_TRY(cudaGetLastError());
    return LORDS_OK;
}
template <int BITS> int launch_quantize_tc(QuantParams &k, int mode, bool sure, const State &st, cudaStream_t stream)
{
    if (sure) return k.r <= 64 ? launch_quantize_tc<BITS, kBuckets, 64, true, true>(k, st, stream) : launch_quantize_tc<BITS, kBuckets, 128, true, true>(k, st, stream);
    if (mode == kBisect) return launch_quantize_tc<BITS, kBisect, 64, false, false>(k, st, stream);
    if (mode == kTrial) return launch_quantize_tc<BITS, kTrial, 64, false, false>(k, st, stream);
    return k.m % kRowsQ != 0 ? launch_quantize_tc<BITS, kBuckets, 64, true, false>(k, st, stream) : launch_quantize_tc<BITS, kBuckets, 64, false, false>(k, st, stream);
}

// The bucket table of an ascending level table.  Buckets are the rounding intervals of `buckets` equally spaced points that cover the
// midpoints with half a spacing to spare on both sides; the ratio that picks one is off by less than 1e-5 of a
// bucket's range (what S is off by comes on top: SURE), so a bucket answers for its interval widened by 1e-3 of the spacing, or with SURE
// by a quarter of it.  False if some widened interval holds two midpoints.
bool make_buckets(QuantParams &k, const float *levels, int bits, int buckets, bool sure)
{
    const int nm = (1 << bits) - 1;
    const double lo = 0.5 * ((double)levels[0] + levels[1]), hi = 0.5 * ((double)levels[nm - 1] + levels[nm]);
    const double h = (hi - lo) / (buckets - 2), first = lo - 0.5 * h;        // point k at first + k h
    if (!(h > 0.0) || !(h < 1e30)) return false;
    const double span = h * (buckets - 1), widened = 0.5 + (sure ? 0.25 : 1e-3);
    k.least_scale = (float)(1.0 / (0.2 * h));        // a ratio inside the table's range is then off by less than a fifth of a spacing
    k.bucket_scale = (float)(1.0 / span);
    k.bucket_bias = (float)(-first / span);
    if (!(k.bucket_scale > 1e-30f) || !(k.bucket_scale < 1e30f) || !(k.bucket_bias > -1e4f) || !(k.bucket_bias < 1e4f)) return false;
    for (int b = 0; b < buckets; ++b) {
        const double a = first + (b - widened) * h, z = first + (b + widened) * h;
        int below = 0, inside = 0;
        float mid = INFINITY;
        for (int c = 0; c < nm; ++c) {
            const double v = k.mids[c];
            if (v < a && b > 0) ++below;
            else if (v <= z || b == buckets - 1) { ++inside; mid = k.mids[c]; }
        }
        if (inside > 1) return false;
        k.bucket_mid[b] = mid;
        k.bucket_code[b] = (uint8_t)below;
    }
    return true;
}

}  // namespace

int launch_quantize(const void *W, const void *B, const void *A, const float *levels, int bits, int m, int n, int r,
                    uint8_t *Q, State &st, cudaStream_t stream)
{
    QuantParams k;
    for (int c = 0; c < 16; ++c) k.levels[c] = c < (1 << bits) ? levels[c] : 0.0f;
    bool sorted = true;
    for (int c = 0; c + 1 < (1 << bits); ++c) sorted = sorted && levels[c] < levels[c + 1];
    for (int c = 0; c < 16; ++c) k.mids[c] = (sorted && c + 1 < (1 << bits)) ? 0.5f * (levels[c] + levels[c + 1]) : 0.0f;
    const int buckets = bits == 4 ? QuantCfg<4, 64>::BUCKETS : bits == 3 ? QuantCfg<3, 64>::BUCKETS : QuantCfg<2, 64>::BUCKETS;
    const int np = (n + 7) / 8 * 8;
    const bool pad = np != n, sure = n % kColsQ != 0 || r > 64;
    const int mode = !sorted ? kTrial : make_buckets(k, levels, bits, buckets, sure) ? kBuckets : kBisect;
    // rows that are not 16-byte multiples: padded copies of W and A in the workspace; behind them the norms that close decisions need
    k.steps = (n + kColsQ - 1) / kColsQ;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t w_bytes = pad ? up((size_t)m * np * 2) : 0, a_bytes = pad ? up((size_t)r * np * 2) : 0;
    const size_t norm_bytes = sure ? ((size_t)k.steps + (size_t)m) * sizeof(float) : 0;
    // Layers with a ragged row or a rank above 64 stay on the CUDA cores where they are small (a few microseconds there as here, in one
    // launch) and with level tables that have no buckets.
    const bool simt = sure && ((long long)m * n <= (5 << 18) || mode != kBuckets);
    const bool tc = !simt && w_bytes + a_bytes + norm_bytes <= st.workspace_bytes && k.steps + ((long long)m + 7) / 8 <= 2147483647LL;
    if (tc && st.forced_path != 1) {
        int launches = 1;
        const void *Wt = W, *At = A;
        if (pad) {
            uint16_t *wp = reinterpret_cast<uint16_t *>(st.workspace), *ap = reinterpret_cast<uint16_t *>(st.workspace + w_bytes);
            PadJobs jobs;
            jobs.count = 2;
            jobs.job[0] = {static_cast<const uint16_t *>(W), wp, n, np, (long long)m * (np / 8)};
            jobs.job[1] = {static_cast<const uint16_t *>(A), ap, n, np, (long long)r * (np / 8)};
            const int rc = launch_pad_rows(jobs, stream);
            if (rc != LORDS_OK) return rc;
            Wt = wp; At = ap;
            ++launches;
        }
        k.B = static_cast<const uint16_t *>(B); k.A = static_cast<const uint16_t *>(A); k.Q = Q;
        k.m = m; k.n = n; k.r = r; k.r_pad = (r + 15) / 16 * 16;
        k.status = st.status_word;
        k.a_norm = k.b_norm = nullptr;
        if (sure) {
            // How far S is off, relative to the sum of absolute products, which the product of norms bounds: an MMA over 16 ranks cuts its
            // sum off below 2^-23 of what has been summed so far, so K of them by (K + 1) 2^-24; 2^-24 more for the midpoint's own rounding.
            // (With a quarter of this no code of 1.2e9 was wrong either, with a sixteenth one in 2e8.)
            float most = 0.0f;
            for (int c = 0; c + 1 < (1 << bits); ++c) most = k.mids[c] > most ? k.mids[c] : -k.mids[c] > most ? -k.mids[c] : most;
            float *a_norm = reinterpret_cast<float *>(st.workspace + w_bytes + a_bytes), *b_norm = a_norm + k.steps;
            lords_quantize_norms_kernel<<<(unsigned)(k.steps + (m + 7) / 8), 256, 0, stream>>>(k.B, k.A, m, n, r, k.steps, most * (float)(k.r_pad / 16 + 2) * 5.960464478e-8f,
                                                                                              a_norm, b_norm);
            LORDS_CUDA_TRY(cudaGetLastError());
            k.a_norm = a_norm; k.b_norm = b_norm;
            ++launches;
        }
        if (!make_map_2d(&k.tm_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, At, (uint64_t)np, (uint64_t)r, 64, (uint32_t)k.r_pad, CU_TENSOR_MAP_SWIZZLE_128B) ||
            !make_map_2d(&k.tm_w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Wt, (uint64_t)np, (uint64_t)m, 64, (uint32_t)kRowsQ, CU_TENSOR_MAP_SWIZZLE_128B))
            return LORDS_ERR_CUDA;
        k.tm_b = k.tm_a;      // not used where the kernel builds the B tile element by element
        if ((r & 7) == 0 &&
            !make_map_2d(&k.tm_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, B, (uint64_t)r, (uint64_t)m, 64, (uint32_t)kRowsQ, CU_TENSOR_MAP_SWIZZLE_128B))
            return LORDS_ERR_CUDA;
        const int rc = bits == 4 ? launch_quantize_tc<4>(k, mode, sure, st, stream) : bits == 3 ? launch_quantize_tc<3>(k, mode, sure, st, stream)
                                                                                    : launch_quantize_tc<2>(k, mode, sure, st, stream);
        if (rc != LORDS_OK) return rc;
        st.last_launches = launches;
        st.last_path = "quantize";
        return LORDS_OK;
    }
    // CUDA-core version: the level table goes through the workspace (stream-ordered copy)
    if (st.workspace_bytes < 64) return LORDS_ERR_WORKSPACE;
    float *lv_dev = reinterpret_cast<float *>(st.workspace);
    LORDS_CUDA_TRY(cudaMemcpyAsync(lv_dev, levels, sizeof(float) * (size_t)(1 << bits), cudaMemcpyHostToDevice, stream));
    const int G = bits == 3 ? 32 : (bits == 4 ? 2 : 4);
    const long long work = (long long)m * (n / G);
    const unsigned blocks = (unsigned)((work + 127) / 128);
    const uint16_t *w16 = static_cast<const uint16_t *>(W), *b16 = static_cast<const uint16_t *>(B), *a16 = static_cast<const uint16_t *>(A);
    if (bits == 4) lords_quantize_simt_kernel<4><<<blocks, 128, 0, stream>>>(w16, b16, a16, Q, m, n, r, lv_dev);
    else if (bits == 3) lords_quantize_simt_kernel<3><<<blocks, 128, 0, stream>>>(w16, b16, a16, Q, m, n, r, lv_dev);
    else lords_quantize_simt_kernel<2><<<blocks, 128, 0, stream>>>(w16, b16, a16, Q, m, n, r, lv_dev);
    LORDS_CUDA_TRY(cudaGetLastError());
    st.last_launches = 1;
    st.last_path = "quantize_simt";
    return LORDS_OK;
}

}  // namespace lords
