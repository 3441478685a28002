// Wide-rank path (65 <= r <= 128) for up to 16 tokens: the scale tile comes from tcgen05, W^ = L[Q] (.) (BA) is formed in the
// registers of the warp that multiplies it.
//
// Per strip of 128 columns one thread issues the scale MMAs  S[128 x 128] = B_tile * A[:, strip]  (Eq. 3; bf16 operands from
// shared memory, fp32 in TMEM).  A consumer warp reads its part of S from TMEM in the accumulator layout of the
// warp-level MMA, multiplies by the levels of the codes (lane-private table) and feeds the products straight to
// mma.sync as the left operand against the activations: that layout is the operand layout, so nothing of W^ is
// written anywhere.  TMEM holds nothing but a ring of two S strips.
//
// Layers of these ranks are computed in 32 bits, as on the CUDA cores: S, the levels and W^ are fp32, W^ enters the product as three
// bf16 parts, x as it is (see split_weights).  Tensor cores cut sums off instead of rounding them, so S of either 64 ranks and the
// first parts' products of every 16 columns start from zero and are added on the CUDA cores; the lower parts' products, 2^-8 of the
// sum, keep to the tensor cores.  Error of the fp32 sums against 64 bits, norms, normal activations, 4096 columns and
// more: 9e-8 to 1.4e-7 (CUDA cores 1.2e-7 to 1.6e-7; W^ and x rounded to fp16 3e-4).
//
// Why a kernel of its own: the factor strip of 128 ranks is 32 KB, which the level table and the rings of the 16-token
// decode kernel leave no room for, and at 128 ranks the scale product outweighs everything else, so it belongs on
// tcgen05: with S by warp-level MMAs (the direct kernel) every warp reads the whole factor strip from shared memory
// again.  4096 x 4096, r = 128, 16 tokens: CUDA cores 585 us, direct kernel 31 us, this kernel 17.5 us (10.4 with W^ in fp16).
//
// CTA: 128 rows; sixteen consumer warps (32 rows and 32 columns of the strip each), a TMA producer, a warp that makes the copy of the
// activations without infinities and NaNs, and a scale issuer.  A cluster shares one row tile and splits its strips; every warp
// sends its partial sums to the CTA that owns the row (asynchronous stores counted on that CTA's barrier), which
// adds them in a fixed order: deterministic, no atomics, no trip through global memory.
//
// Bound: the consumers' instructions (13.7 a weight: look-up, product, cutting into parts, MMAs) and the latency of their chain, four
// warps to a scheduler: 1.6 us a strip of 16384 weights (8192 columns, eight more strips a CTA, take 12.4 us more), beside which the strip's
// arrival (44 KB from L2, about a third of that time) and its scale MMAs (a sixth) run.
//
// Every wait is bounded; on expiry the role records LORDS_ERR_TIMEOUT and leaves its loop.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lords_internal.h"
#include "lords_ptx.cuh"
#include "lords_tc_common.cuh"
#include "lords_warp_mma.cuh"

namespace lords {

namespace {

using namespace ptx;

constexpr int kRows = 128;                          // rows of W^ per CTA = UMMA M
constexpr int kStrip = 128;                         // columns per strip
constexpr int kConsumers = 16;
constexpr int kSplit = 4;                           // warps that share a row group of 32: a quarter of the strip's columns each
constexpr int kTmaWarp = kConsumers, kConvWarp = kConsumers + 1, kScaleWarp = kConsumers + 2;
constexpr int kThreads = (kConsumers + 3) * 32;
constexpr int kClusterMax = 16;
constexpr int DS = 2;                               // S strips in TMEM
constexpr uint32_t kTmemCols = DS * 2 * kStrip;     // S of ranks 0 .. 63 and of the others, apart
constexpr int kRankMax = 128;
constexpr int kAAtom = kRankMax * 128;              // 64 columns of the factor strip, 128-byte swizzle
constexpr int kBAtom = kRows * 128;                 // B[128 x 64 ranks], K-major, 128-byte swizzle; two of them

// BITS: code width.  TG: tokens in groups of eight (zero padded).
template <int BITS, int TG> struct WideCfg {
    static constexpr int ENTRIES = 1 << 2 * BITS;                             // level pairs
    static constexpr int LUT = ENTRIES * 128;                                 // 16 copies of every pair in fp32, one for a lane of each half warp
    static constexpr int QROW = kStrip * BITS / 8;                            // 64 / 48 / 32 bytes
    static constexpr int QTILE = kRows * QROW;
    static constexpr int XATOM = TG * 8 * 128;                                // 64 columns of the activations, 128-byte swizzle
    static constexpr int XTILE = 2 * XATOM;
    static constexpr int RED = (kRows + kClusterMax) * TG * 8 * 4;            // partial sums received: cluster x rows owned x tokens
    static constexpr int FIXED = 1024 + 2 * kBAtom + LUT + RED + 512;
    static constexpr int STAGE = 2 * kAAtom + QTILE + 2 * XTILE;              // the activations as they are and without infinities and NaNs
    static constexpr int D = (232448 - FIXED) / STAGE < 4 ? (232448 - FIXED) / STAGE : 4;    // strips in flight
    static constexpr int SMEM = FIXED + D * STAGE;
    static_assert(D >= 2 && QTILE % 1024 == 0 && XATOM % 1024 == 0, "swizzled tiles start on their pattern's boundary");
};

struct alignas(64) WideParams {
    CUtensorMap tm_q;     // u8 [m][n*bits/8], box {QROW, 128}; swizzle 64 / none / 32 bytes for 4 / 3 / 2 bits
    CUtensorMap tm_a;     // bf16 [r][n], box {64, r_pad}, 128-byte swizzle (ranks past r and columns past n read as zero)
    CUtensorMap tm_x;     // bf16 [M][n], box {64, TG * 8}, 128-byte swizzle (tokens past M read as zero)
    CUtensorMap tm_b;     // bf16 [m][r], box {64, 128}, 128-byte swizzle; used if rows of B are 16-byte multiples
    const uint16_t *B;    // bf16 [m][r]
    float levels[16];
    int M, m, n, r, r_pad;
    int strips;           // strips per row
    int per_rank;         // rows of the tile that one CTA of the cluster adds up: ceil(128 / cluster)
    uint32_t per_rank_inv;   // ceil(65536 / per_rank): row / per_rank by a multiplication
    void *y;
    int y_f32;
    int *status;
};

// Byte offset of 32-column group c (0..3) of row `row` in a code tile as the tensor-map copy lays it out: 4-bit rows are 64
// bytes with 16-byte chunks swizzled over four, 2-bit rows 32 bytes (a group is 8 bytes) with chunks swapped
// every four rows, 3-bit rows 48 bytes as they are; eight consecutive rows fall into different banks.
template <int BITS> __device__ __forceinline__ uint32_t code_offset(int row, int c)
{
    if constexpr (BITS == 4) return (uint32_t)(row * 64 + ((c ^ ((row >> 1) & 3)) << 4));
    else if constexpr (BITS == 3) return (uint32_t)(row * 48 + c * 12);
    else return (uint32_t)(row * 32 + (((c >> 1) ^ ((row >> 2) & 1)) << 4) + (c & 1) * 8);
}

__device__ __forceinline__ uint64_t pair_at(const uint32_t (&v)[16], int e) { return f32x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])); }

template <int BITS, int TG>
__global__ void __launch_bounds__(kThreads, 1) lords_wide_kernel(const __grid_constant__ WideParams p)
{
    using C = WideCfg<BITS, TG>;
    constexpr int D = C::D, MT = TG * 8;
    extern __shared__ uint8_t wide_smem[];
    const uint32_t b_tile = (smem_u32(wide_smem) + 1023u) & ~1023u;
    const uint32_t a_s = b_tile + 2 * kBAtom, q_s = a_s + D * 2 * kAAtom, x_s = q_s + D * C::QTILE, lut = x_s + D * 2 * C::XTILE;
    const uint32_t red = lut + C::LUT, bars = red + C::RED;
    const uint32_t bar_q = bars, bar_x = bar_q + 8 * D, bar_free = bar_x + 8 * D;              // bar_q: codes and activations have landed
    const uint32_t bar_a = bar_free + 8 * D, bar_a_free = bar_a + 8 * D, bar_s = bar_a_free + 8 * D, bar_s_free = bar_s + 8 * DS;
    const uint32_t bar_b = bar_s_free + 8 * DS, bar_red = bar_b + 8, tmem_slot = bar_red + 8;
    static_assert(8 * (5 * D + 2 * DS + 2) + 4 <= 512, "barrier area");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    const int csize = (int)cluster_nctarank(), rank = (int)cluster_ctarank();
    const int row0 = ((int)blockIdx.x / csize) * kRows;
    const int s_a = rank * p.strips / csize, total = (rank + 1) * p.strips / csize - s_a;
    const int own0 = rank * p.per_rank, own_n = own0 >= kRows ? 0 : (own0 + p.per_rank < kRows ? p.per_rank : kRows - own0);
    const bool b_by_tma = (p.r & 7) == 0;
    const int *status = p.status;
    bool failed = false;

    if (warp == kTmaWarp) {
        // ------------------------------------------------------------------ producer: barriers, weights, activations
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < D; ++k) {
                mbar_init(bar_q + 8 * k, 2);
                mbar_init(bar_x + 8 * k, 1);
                mbar_init(bar_free + 8 * k, kConsumers);
                mbar_init(bar_a + 8 * k, 1);
                mbar_init(bar_a_free + 8 * k, 1);
            }
#pragma unroll
            for (int k = 0; k < DS; ++k) { mbar_init(bar_s + 8 * k, 1); mbar_init(bar_s_free + 8 * k, kConsumers); }
            mbar_init(bar_b, 1);
            mbar_init(bar_red, 1);
            fence_mbar_init();
            // the partial sums this CTA will receive: every pair of tokens that exists, of its rows, from every CTA
            mbar_expect_tx(bar_red, (uint32_t)(csize * own_n * ((p.M + 1) / 2) * 8));
        }
        __syncwarp();
        // these ranks are stream-ordered calls: no weight is read before the previous launch has ended
        asm volatile("bar.arrive 1, %0;" ::"n"(kThreads) : "memory");          // the barriers exist
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // waited for before the first remote store
        griddep_launch_dependents();
        griddep_wait();
        auto factors = [&](int it) {
            const uint32_t bar = bar_a + 8 * (it % D), dst = a_s + (uint32_t)((it % D) * 2 * kAAtom);
            mbar_expect_tx(bar, (uint32_t)(2 * p.r_pad * 128));
            tma_load_2d(dst, &p.tm_a, (s_a + it) * kStrip, 0, bar);
            tma_load_2d(dst + kAAtom, &p.tm_a, (s_a + it) * kStrip + 64, 0, bar);
        };
        auto codes = [&](int it) {
            const uint32_t bar = bar_q + 8 * (it % D);
            mbar_expect_tx(bar, (uint32_t)C::QTILE);
            tma_load_2d(q_s + (uint32_t)((it % D) * C::QTILE), &p.tm_q, (s_a + it) * C::QROW, row0, bar);
        };
        auto activations = [&](int it) {
            const uint32_t bar = bar_q + 8 * (it % D);
            const uint32_t dst = x_s + (uint32_t)((it % D) * 2 * C::XTILE);
            mbar_expect_tx(bar, (uint32_t)C::XTILE);
            tma_load_2d(dst, &p.tm_x, (s_a + it) * kStrip, 0, bar);
            tma_load_2d(dst + C::XATOM, &p.tm_x, (s_a + it) * kStrip + 64, 0, bar);
        };
        if (lane == 0) {
            if (b_by_tma) {
                mbar_expect_tx(bar_b, (uint32_t)(2 * kBAtom));
                tma_load_2d(b_tile, &p.tm_b, 0, row0, bar_b);
                tma_load_2d(b_tile + kBAtom, &p.tm_b, 64, row0, bar_b);
            }
            for (int it = 0; it < D && it < total; ++it) {
                factors(it);
                codes(it);
                activations(it);
            }
            for (int it = D; it < total; ++it) {
                if (!mbar_wait(bar_a_free + 8 * (it % D), (uint32_t)((it / D - 1) & 1), status, 76)) { failed = true; break; }
                factors(it);
                if (!mbar_wait(bar_free + 8 * (it % D), (uint32_t)((it / D - 1) & 1), status, 71)) { failed = true; break; }
                codes(it);
                activations(it);
            }
        }
        __syncwarp();
    } else if (warp == kConvWarp) {
        // ------------------------------------------------------------------ the second copy of the activations, word by word wherever the swizzle put it
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        griddep_launch_dependents();
        griddep_wait();
        for (int it = 0; it < total; ++it) {
            const int st = it % D;
            if (!mbar_wait_warp(bar_q + 8 * st, (uint32_t)((it / D) & 1), status, 75)) { failed = true; break; }
            // all loads first: one after the other's store, each would wait for the way through shared memory
            const uint32_t base = x_s + (uint32_t)(st * 2 * C::XTILE + lane * 16);
            uint4 v[MT / 2];
#pragma unroll
            for (int k = 0; k < MT / 2; ++k) v[k] = lds_v4(base + (uint32_t)(k * 512));
#pragma unroll
            for (int k = 0; k < MT / 2; ++k)
                sts_v4(base + (uint32_t)(C::XTILE + k * 512), make_uint4(finite_pair(v[k].x), finite_pair(v[k].y), finite_pair(v[k].z), finite_pair(v[k].w)));
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_x + 8 * st);
        }
    } else if (warp == kScaleWarp) {
        // ------------------------------------------------------------------ scale MMAs: S of strip `it` into TMEM strip it % DS
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
        tc_fence_before_sync();
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
        tc_fence_after_sync();
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        griddep_launch_dependents();
        griddep_wait();
        uint32_t tmem_base;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));
        tmem_base = warp_uniform(tmem_base);
        const uint32_t leader = elect_one();
        constexpr uint32_t idesc = umma_idesc_f16(1, 0, 1, kRows, kStrip);     // bf16, B operand MN-major
        const uint32_t desc_hi = (uint32_t)(umma_desc_sw128(0, 1024, 16) >> 32);
        const uint32_t b_lo = (uint32_t)umma_desc_sw128(0, 1024, 16) | ((b_tile & 0x3FFFFu) >> 4);
        const uint32_t a_lo0 = (uint32_t)umma_desc_sw128(0, 1024, (uint32_t)kAAtom) | ((a_s & 0x3FFFFu) >> 4);
        const int rsteps = p.r_pad / 16;
        if (b_by_tma && !mbar_wait_warp(bar_b, 0, status, 77)) failed = true;
        for (int it = 0; it < total && !failed; ++it) {
            const int sa = it % D, sd = it % DS;
            // Up to eight tokens this wait sleeps between tries: without, layers were up to 7 % slower (5646 x 512, 2 bits, rank 71, two tokens:
            // 9.7 us and 10.4; 72 layers 1.0 % on average).  With more tokens it costs 0.3 % (4096 x 4096, rank 128, 16 tokens: 17.5 us, 17.3 without).
            if (!mbar_wait_warp2<TG == 1 ? kWaitSleepNs : 0>(bar_a + 8 * sa, (uint32_t)((it / D) & 1), bar_s_free + 8 * sd,
                                                            (uint32_t)((it / DS + 1) & 1), status, 78)) { failed = true; break; }
            tc_fence_after_sync();
            const uint32_t a_lo = a_lo0 + (uint32_t)(sa * ((2 * kAAtom) >> 4));
            for (int k = 0; k < rsteps; ++k)                                   // 64 ranks per atom of the B tile, and per sum
                umma_f16_ss(tmem_base + (uint32_t)((2 * sd + (k >> 2)) * kStrip), umma_desc_pack(b_lo + (k >> 2) * (kBAtom >> 4) + (k & 3) * 2, desc_hi),
                            umma_desc_pack(a_lo + k * 128, desc_hi), idesc, (k & 3) > 0, leader);
            umma_commit(bar_s + 8 * sd, leader);
            umma_commit(bar_a_free + 8 * sa, leader);
        }
        // no commit is still on its way to a barrier when the CTA ends
        if (!failed && total > 0 && !mbar_wait_warp(bar_a_free + 8 * ((total - 1) % D), (uint32_t)(((total - 1) / D) & 1), status, 80)) failed = true;
    } else {
        // ------------------------------------------------------------------ consumers
        // row group rw (its TMEM quadrant), column quarter ch
        const int g = lane >> 2, t = lane & 3, rw = warp & 3, ch = warp >> 2;
        fill_pair_table<BITS, false>(lut, p.levels, tid);
        if (!b_by_tma) {
            // rows of B that are not 16-byte multiples: element by element, zeros past rank r and past row m
            griddep_wait();
            const int rr = tid >> 2, i = row0 + rr;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int chunk = (tid & 3) * 4 + c;                           // of the row's sixteen
                uint32_t w4[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) w4[e] = load_b_pair(p.B, i, chunk * 8 + e * 2, p.m, p.r);
                sts_v4(b_tile + (uint32_t)((chunk >> 3) * kBAtom + (rr >> 3) * 1024 + (rr & 7) * 128 + (((chunk & 7) ^ (rr & 7)) * 16)),
                       make_uint4(w4[0], w4[1], w4[2], w4[3]));
            }
            fence_proxy_async_smem();
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");            // table, B tile, barriers and TMEM are in place
        tc_fence_after_sync();
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        griddep_launch_dependents();
        griddep_wait();
        uint32_t tmem_base;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));

        float acc[2][TG][4], low[2][TG][4];                                    // low: the sums of the weights' lower parts
#pragma unroll
        for (int rg = 0; rg < 2; ++rg)
#pragma unroll
            for (int k = 0; k < TG; ++k) {
                acc[rg][k][0] = acc[rg][k][1] = acc[rg][k][2] = acc[rg][k][3] = 0.0f;
                low[rg][k][0] = low[rg][k][1] = low[rg][k][2] = low[rg][k][3] = 0.0f;
            }
        const uint32_t lut_lane = lut + 8u * (uint32_t)(lane & 15);
        // x, 16 columns at a time: token row lane & 7 of group lane >> 4, 16-byte chunk lane >> 3 & 1 (the next 16 columns are two chunks
        // on, bit 5 of the address), chunks swizzled by the row
        const uint32_t x_lane = x_s + (uint32_t)((ch >> 1) * C::XATOM + (TG == 2 ? (lane >> 4) * 1024 : 0) + (lane & 7) * 128 +
                                                 (((((ch & 1) * 4) + ((lane >> 3) & 1)) ^ (lane & 7)) << 4));
        const uint32_t s_lane = tmem_base + ((uint32_t)(rw * 32) << 16) + (uint32_t)(ch * 32);

        for (int it = 0; it < total; ++it) {
            const int st = it % D, sd = it % DS;
            if (!mbar_wait_warp3(bar_s + 8 * sd, (uint32_t)((it / DS) & 1), bar_q + 8 * st, (uint32_t)((it / D) & 1),
                                 bar_x + 8 * st, (uint32_t)((it / D) & 1), true, status, 72)) { failed = true; break; }
            tc_fence_after_sync();
            const uint32_t q_tile = q_s + (uint32_t)(st * C::QTILE), x_tile = x_lane + (uint32_t)(st * 2 * C::XTILE);
#pragma unroll
            for (int rg = 0; rg < 2; ++rg) {                                   // units of 16 rows x 32 columns
                uint32_t u[16], v[16];
                const uint32_t at = s_lane + ((uint32_t)(rg * 16) << 16) + (uint32_t)(2 * sd * kStrip);
                tmem_ld_16x32_frag(at, u);
                tmem_ld_16x32_frag(at + kStrip, v);
                CodeWords<BITS> w0, w1;
                w0.read(q_tile + code_offset<BITS>(rw * 32 + rg * 16 + g, ch));
                w1.read(q_tile + code_offset<BITS>(rw * 32 + rg * 16 + g + 8, ch));
                tmem_wait_ld(u);
                tmem_wait_ld(v);
                uint64_t s[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) s[e] = f32x2_add(pair_at(u, e), pair_at(v, e));
                if (rg == 1) {
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_s_free + 8 * sd);         // S is in registers: the next one may be written
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint64_t w[4] = {w0.weights(2 * h, t, lut_lane, s[4 * h]), w1.weights(2 * h, t, lut_lane, s[4 * h + 1]),
                                           w0.weights(2 * h + 1, t, lut_lane, s[4 * h + 2]), w1.weights(2 * h + 1, t, lut_lane, s[4 * h + 3])};
                    uint32_t hi[4], mid[4], lo[4];
                    split_weights(w, hi, mid, lo);
                    uint32_t xb[2 * TG], xf[2 * TG];
                    if constexpr (TG == 2) {
                        ldmatrix_x4(x_tile ^ (uint32_t)(h * 32), xb);
                        ldmatrix_x4((x_tile ^ (uint32_t)(h * 32)) + C::XTILE, xf);
                    } else {
                        ldmatrix_x2(x_tile ^ (uint32_t)(h * 32), xb);
                        ldmatrix_x2((x_tile ^ (uint32_t)(h * 32)) + C::XTILE, xf);
                    }
#pragma unroll
                    for (int k = 0; k < TG; ++k) {
                        add_mma_bf16(acc[rg][k], hi, xb[2 * k], xb[2 * k + 1]);
                        mma_bf16(low[rg][k], mid, xf[2 * k], xf[2 * k + 1]);
                        mma_bf16(low[rg][k], lo, xf[2 * k], xf[2 * k + 1]);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_free + 8 * st);
        }

#pragma unroll
        for (int k = 0; k < 2 * TG; ++k) add_low(acc[k / TG][k % TG], low[k / TG][k % TG]);

        // The four column quarters of a row group meet first, in the factor ring (every copy into it and every MMA on it has
        // completed: the last strip's S has been waited for), so that one partial sum per row and token goes out.
        const uint32_t park = a_s + (uint32_t)(rw * 32 * MT * 4 + lane * 16);       // [quarter - 1][row group][value][lane]
        asm volatile("bar.sync 2, %0;" ::"n"(kConsumers * 32) : "memory");
        if (ch > 0) {
#pragma unroll
            for (int k = 0; k < 2 * TG; ++k)
                sts_v4(park + (uint32_t)((ch - 1) * kRows * MT * 4 + k * 512),
                       make_uint4(__float_as_uint(acc[k / TG][k % TG][0]), __float_as_uint(acc[k / TG][k % TG][1]), __float_as_uint(acc[k / TG][k % TG][2]),
                                  __float_as_uint(acc[k / TG][k % TG][3])));
        }
        asm volatile("bar.sync 2, %0;" ::"n"(kConsumers * 32) : "memory");
        // partial sums to the CTA that owns the row; a CTA that gave up still sends (what it has), so nobody waits in vain
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (ch == 0) {
#pragma unroll
            for (int c = 0; c < kSplit - 1; ++c)
#pragma unroll
                for (int k = 0; k < 2 * TG; ++k) {
                    const uint4 v = lds_v4(park + (uint32_t)(c * kRows * MT * 4 + k * 512));
                    acc[k / TG][k % TG][0] += __uint_as_float(v.x);
                    acc[k / TG][k % TG][1] += __uint_as_float(v.y);
                    acc[k / TG][k % TG][2] += __uint_as_float(v.z);
                    acc[k / TG][k % TG][3] += __uint_as_float(v.w);
                }
#pragma unroll
            for (int rg = 0; rg < 2; ++rg)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int row = rw * 32 + rg * 16 + g + 8 * h, owner = (int)(((uint32_t)row * p.per_rank_inv) >> 16);
                    const uint32_t dst = map_to_rank(red + (uint32_t)(((rank * p.per_rank + row - owner * p.per_rank) * MT + 2 * t) * 4), (uint32_t)owner);
                    const uint32_t dbar = map_to_rank(bar_red, (uint32_t)owner);
#pragma unroll
                    for (int k = 0; k < TG; ++k)
                        if (k * 8 + 2 * t < p.M) st_async_cluster_2f32(dst + (uint32_t)(k * 32), acc[rg][k][2 * h], acc[rg][k][2 * h + 1], dbar);
                }
        }
        if (own_n > 0) {
            if (!mbar_wait_cluster(bar_red, 0, status, 74)) failed = true;
            else
                for (int e = warp, groups = (own_n + 31) / 32; e < p.M * groups; e += kConsumers) {
                    const int tok = e / groups, row = (e - tok * groups) * 32 + lane, i = row0 + own0 + row;
                    if (row < own_n) {
                        float sum = 0.0f;
                        for (int rr = 0; rr < csize; ++rr)
                            sum += __uint_as_float(lds_u32(red + (uint32_t)(((rr * p.per_rank + row) * MT + tok) * 4)));
                        if (i < p.m) store_out(p.y, p.y_f32, (size_t)tok * p.m + i, sum);
                    }
                }
        }
    }
    if (failed) ptx::record_give_up(p.status, LORDS_ERR_TIMEOUT);
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kScaleWarp) {
        tc_fence_after_sync();
        uint32_t tmem_base;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));
        tmem_dealloc(tmem_base, kTmemCols);
    }
    // no CTA leaves while stores of its own may be on their way to another (the last three warps have not waited on the
    // first phase of the cluster barrier yet)
    if (warp >= kConsumers) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

template <int BITS, int TG> struct WideVariant {
    using C = WideCfg<BITS, TG>;
    static void fill(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int cs, int tiles, cudaStream_t stream)
    {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg = cudaLaunchConfig_t{};
        cfg.gridDim = dim3((unsigned)(tiles * cs));
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = C::SMEM;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
    }
    // Clusters of `cs` CTAs that can be resident at once (0: such a cluster cannot run).
    static int max_clusters(int dev, int cs)
    {
        static int cache[kMaxDevices][kClusterMax + 1];   // 0 = not asked yet, -1 = cannot run
        if (cache[dev][cs] == 0) {
            auto kernel = lords_wide_kernel<BITS, TG>;
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr[2];
            fill(cfg, attr, cs, 1, nullptr);
            int n = 0;
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess ||
                cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess)
                (void)cudaGetLastError();
            cache[dev][cs] = n >= 1 ? n : -1;
        }
        return cache[dev][cs] > 0 ? cache[dev][cs] : 0;
    }
    static int launch(WideParams &k, const Problem &p, State &st, cudaStream_t stream)
    {
        const int dev = device_slot(st), tiles = (p.m + kRows - 1) / kRows, lim = kClusterMax < k.strips ? kClusterMax : k.strips;
        int cs = 0;
        if (st.forced_splitk > 0) {
            for (cs = st.forced_splitk < lim ? st.forced_splitk : lim; cs > 1 && max_clusters(dev, cs) == 0;) --cs;
        } else {
            // waves of clusters times (strips of a CTA + a fixed part worth three)
            double best = 1e30;
            for (int c = 1; c <= lim; ++c) {
                const int res = max_clusters(dev, c);
                if (res == 0) continue;
                const double t = (double)((tiles + res - 1) / res) * ((k.strips + c - 1) / c + 3.0);
                if (t <= best) { best = t; cs = c; }
            }
        }
        if (cs < 1 || max_clusters(dev, cs) == 0) return LORDS_ERR_UNSUPPORTED;
        const uint64_t row_bytes = (uint64_t)p.n * BITS / 8;
        k.tm_b = CUtensorMap{};   // not used where the kernel builds the B tile element by element
        if (!make_map_2d(&k.tm_q, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, p.q, row_bytes, (uint64_t)p.m, (uint32_t)C::QROW, (uint32_t)kRows,
                         BITS == 4 ? CU_TENSOR_MAP_SWIZZLE_64B : BITS == 3 ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_32B) ||
            !make_map_2d(&k.tm_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p.A, (uint64_t)p.n, (uint64_t)p.r, 64, (uint32_t)k.r_pad, CU_TENSOR_MAP_SWIZZLE_128B) ||
            !make_map_2d(&k.tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p.x, (uint64_t)p.n, (uint64_t)p.M, 64, (uint32_t)(TG * 8), CU_TENSOR_MAP_SWIZZLE_128B) ||
            ((p.r & 7) == 0 && !make_map_2d(&k.tm_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p.B, (uint64_t)p.r, (uint64_t)p.m, 64, (uint32_t)kRows,
                                            CU_TENSOR_MAP_SWIZZLE_128B)))
            return LORDS_ERR_CUDA;
        k.per_rank = (kRows + cs - 1) / cs;
        k.per_rank_inv = (uint32_t)((65536 + k.per_rank - 1) / k.per_rank);
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[2];
        fill(cfg, attr, cs, tiles, stream);
        if (p.ordered) attr[1].val.programmaticStreamSerializationAllowed = 0;
        LORDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, lords_wide_kernel<BITS, TG>, k));
        return LORDS_OK;
    }
};

template <int BITS> int launch_wide(WideParams &k, const Problem &p, State &st, cudaStream_t stream)
{
    return p.M <= 8 ? WideVariant<BITS, 1>::launch(k, p, st, stream) : WideVariant<BITS, 2>::launch(k, p, st, stream);
}

}  // namespace

// Rules of this path: M <= 16; 64 < r <= 128; n a multiple of 32 (4-bit), 64 (2-bit) or 128 (3-bit), which makes every row
// pitch a multiple of 16 bytes.  Anything else: LORDS_ERR_UNSUPPORTED.
int launch_wide(const Problem &p, State &st, cudaStream_t stream)
{
    if (p.M > 16 || p.r <= 64 || p.r > kRankMax || p.n % (p.bits == 4 ? 32 : p.bits == 2 ? 64 : 128) != 0) return LORDS_ERR_UNSUPPORTED;
    WideParams k;
    k.B = p.B;
    for (int c = 0; c < 16; ++c) k.levels[c] = p.levels[c];
    k.M = p.M; k.m = p.m; k.n = p.n; k.r = p.r;
    k.r_pad = (p.r + 15) / 16 * 16;
    k.strips = (p.n + kStrip - 1) / kStrip;
    k.y = p.y; k.y_f32 = p.y_f32;
    k.status = st.status_word;
    const int rc = p.bits == 4 ? launch_wide<4>(k, p, st, stream) : p.bits == 3 ? launch_wide<3>(k, p, st, stream) : launch_wide<2>(k, p, st, stream);
    if (rc != LORDS_OK) return rc;
    st.last_launches = 1;
    st.last_path = "wide";
    return LORDS_OK;
}

}  // namespace lords
