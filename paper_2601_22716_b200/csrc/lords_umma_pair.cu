// Scale-MMA path for large calls (lords_umma.cu has the rule): the schedule of lords_umma.cu on CTA pairs (cta_group::2).
//
// What bounds the single-CTA kernel at these sizes is the way from L2 into shared memory: 40 KB per 64-column step and SM, about 40
// bytes a clock, which is also where a plain product with 256 x 256 pair tiles stands (32 KB a step).  Here a pair of CTAs owns 256
// rows of W^ and up to 256 tokens; each CTA holds half of the tokens' activations, rebuilds its own 128 rows of W^ in TMEM
// and loads half of the factor tiles: 22 KB per step and SM, most of it activations.  Calls with their pre-passes, one CTA per tile
// against pairs, a graph of two or three layers: 4096 x 14336, 2048 tokens 248 us and 206 (239 in longer runs, at the clock that the
// power cap leaves); 14336 x 4096, 512 tokens 79 and 60.
//
// A step is 128 columns (a code stage), two k-steps of 64.  TMEM (512 columns): the accumulator [128 x BN], one buffer of S for a step
// [128 x 128] fp32 and a ring of four W^ k-steps [128 x 64] fp16.  S and W^ are separate so that neither the scale
// MMA nor the look-ups wait for main MMAs: a worker takes S into registers, releases it, and needs the main MMA of four k-steps
// before only when it stores.  Scale MMAs go out ahead of the main MMAs of the step before, so that they execute as soon as those of the step
// before that have finished.
//   warps 0..15  two groups of eight, one per k-step of a step: S -> registers, level pairs, W^ to TMEM; after the last step of a
//                piece: accumulator -> y, or to scratch
//   warp 16      main MMAs (issued by the pair's even CTA): M = 256, N = BN
//   warp 17      scale MMAs (likewise): M = 256, N = 128, 64 columns of A from either CTA
//   warp 18      TMEM; then TMA of the factor tiles and, per piece, of B (both into the even CTA's barriers)
//   warp 19      TMA of activations and codes
// Pairs are persistent; tiles of whole waves run one per pair, the steps of the tiles left over are dealt out evenly
// (lords_pair.cuh), and the pieces of a tile meet in scratch in a fixed order.
//
// Every wait is bounded; on expiry the role records LORDS_ERR_TIMEOUT and leaves its loop.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lords_dequant.cuh"
#include "lords_internal.h"
#include "lords_pair.cuh"
#include "lords_ptx.cuh"
#include "lords_tc_common.cuh"

namespace lords {

namespace {

using namespace ptx;

constexpr int kPRows = 256;                    // rows of W^ per pair
constexpr int kPTok = 256;                     // most tokens per tile
constexpr int kPWorkers = 16;
constexpr int kPIssuer = kPWorkers, kPScale = kPWorkers + 1, kPTmaA = kPWorkers + 2, kPTmaX = kPWorkers + 3;
constexpr int kPThreads = (kPWorkers + 4) * 32;
constexpr uint32_t kPTmemCols = 512, kPSCol = 256, kPWCol = 384;      // accumulator | S of a step | ring of W^ k-steps
constexpr int kPDone = 8;                      // "main MMAs of the k-step done" barriers, by k-step
constexpr int kPW = 4;                         // W^ ring
constexpr int kPSA = 3;                        // factor-tile ring (steps)
constexpr int kPSQ = 4;                        // code ring (steps)

// BITS: code width.  RP: padded rank that the factor tiles are sized for (32 or 64).
template <int BITS, int RP> struct PCfg {
    static constexpr int XTILE = kPTok / 2 * 128;                // this CTA's half of the tokens, 64 columns fp16
    static constexpr int ATILE = RP * 128;                       // 64 columns of A
    static constexpr int BTILE = 128 * 128;
    static constexpr int QROW = 128 * BITS / 8, QSTAGE = 128 * QROW;
    static constexpr int LUT_ENTRIES = BITS == 4 ? 256 : BITS == 3 ? 64 : 16;
    static constexpr int STAGE = 16 * 64;                        // a worker warp's 32 rows x 16 tokens of y
    static constexpr int REST = 1024 + kPSA * ATILE + BTILE + kPSQ * QSTAGE + LUT_ENTRIES * 128 + kPWorkers * STAGE + 512;
    static constexpr int SX = (232448 - REST) / XTILE < kPDone ? (232448 - REST) / XTILE : kPDone;      // activation ring (k-steps): 6 to 8
    static constexpr int SMEM = REST + SX * XTILE;
};

struct alignas(64) PairParams {
    CUtensorMap tm_x;     // fp16 [M][n], box {64, bn / 2}, 128-byte swizzle
    CUtensorMap tm_a;     // bf16 [r][n], box {64, r_pad}, 128-byte swizzle
    CUtensorMap tm_b;     // bf16 [m][r rounded up to 8], box {64, 128}, 128-byte swizzle (zeros past the rank and past row m)
    CUtensorMap tm_q;     // u8 [m][n * bits / 8], box {QROW, 128}
    float levels[16];
    int M, m, r_pad, bn;
    int steps;            // 128-column steps of a tile
    int tok_tiles, tiles, pairs, whole;
    int b_early;          // B is the caller's (not the pre-pass's padded copy)
    float *partial;       // [pair][2][bn / 4][128 rows][4 tokens]: a piece that does not begin its tile
    int *flags;           // [pair][2]: warps that have put their part of the piece into scratch; zero between calls
    void *y;
    int y_f32;
    int *status;
};

template <int BITS, int RP>
__global__ void __launch_bounds__(kPThreads, 1) lords_umma_pair_kernel(const __grid_constant__ PairParams p)
{
    using C = PCfg<BITS, RP>;
    extern __shared__ uint8_t p_smem[];
    const uint32_t x0 = (smem_u32(p_smem) + 1023u) & ~1023u;
    const uint32_t b_tile = x0 + C::SX * C::XTILE, a0 = b_tile + C::BTILE, q0 = a0 + kPSA * C::ATILE, lut = q0 + kPSQ * C::QSTAGE;
    const uint32_t stage0 = lut + C::LUT_ENTRIES * 128, bars = stage0 + kPWorkers * C::STAGE;
    // in the even CTA, for the pair
    const uint32_t bar_x = bars, bar_a = bar_x + 8 * C::SX, bar_w = bar_a + 8 * kPSA, bar_s_free = bar_w + 8 * kPW, bar_b = bar_s_free + 8;
    const uint32_t bar_acc_free = bar_b + 8;
    // in both CTAs: commits arrive at either
    const uint32_t bar_done = bar_acc_free + 8, bar_a_free = bar_done + 8 * kPDone, bar_s = bar_a_free + 8 * kPSA, bar_acc = bar_s + 8;
    const uint32_t bar_q = bar_acc + 8, bar_q_free = bar_q + 8 * kPSQ, tmem_slot = bar_q_free + 8 * kPSQ;
    static_assert(8 * (C::SX + 2 * kPSA + kPW + kPDone + 5 + 2 * kPSQ) + 4 <= 512, "barrier area");

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster_ctarank();
    // Pairs are numbered against the launch order: a pair waits only for pieces of pairs with a lower block index,
    // which the hardware has started before it.
    const int pair = p.pairs - 1 - (int)(blockIdx.x >> 1);
    const int *status = p.status;
    bool failed = false;

    if (warp == kPTmaX) {
        if (lane == 0) {
            for (int k = 0; k < C::SX; ++k) mbar_init(bar_x + 8 * k, 1);
            for (int k = 0; k < kPSA; ++k) { mbar_init(bar_a + 8 * k, 1); mbar_init(bar_a_free + 8 * k, 1); }
            for (int k = 0; k < kPW; ++k) mbar_init(bar_w + 8 * k, kPWorkers);                  // eight warps of either CTA
            mbar_init(bar_s_free, 2 * kPWorkers);
            mbar_init(bar_b, 1);
            mbar_init(bar_acc_free, 2 * kPWorkers);
            for (int k = 0; k < kPDone; ++k) mbar_init(bar_done + 8 * k, 1);
            mbar_init(bar_s, 1);
            mbar_init(bar_acc, 1);
            for (int k = 0; k < kPSQ; ++k) { mbar_init(bar_q + 8 * k, 1); mbar_init(bar_q_free + 8 * k, kPWorkers); }
            fence_mbar_init();
            tma_prefetch_desc(&p.tm_q);
            tma_prefetch_desc(&p.tm_x);
        }
    } else if (warp == kPTmaA) {
        tmem_alloc2(tmem_slot, kPTmemCols);
    } else if (warp < kPWorkers) {
        // level-pair table: word e * 32 + lane is lane's copy of entry e (bank = lane: look-ups never conflict)
#pragma unroll
        for (int e = warp; e < C::LUT_ENTRIES; e += kPWorkers) {
            const __half2 v = __floats2half2_rn(p.levels[e & ((1 << BITS) - 1)], p.levels[e >> BITS]);
            sts_u32(lut + 4u * (uint32_t)(e * 32 + lane), *reinterpret_cast<const uint32_t *>(&v));
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // both CTAs' barriers exist
    tc_fence_after_sync();
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));
    griddep_launch_dependents();

    Schedule sched(p.pairs, p.whole, p.tiles, p.steps, pair);
    Piece w;
    int st = 0;                                   // steps so far, over all pieces: ring positions and phases
    // Every role passes the end of the previous launch before its first bounded wait for something that needs the activations, itself or
    // by way of another role that waits there; what comes before that runs ahead on weights alone.
    bool passed = false;
    auto previous_launch = [&] {
        if (!passed) { griddep_wait(); passed = true; }
    };
    if (warp == kPTmaX) {
        // ------------------------------------------------------------------ activations (this CTA's half of the tokens) and codes
        if (lane == 0) {
            const uint32_t x_pair0 = map_to_rank(bar_x, 0);
            const uint32_t x_tx = (uint32_t)(p.bn * 128);
            while (!failed && sched.next(w)) {
                const int rt = w.tile / p.tok_tiles, tt = w.tile - rt * p.tok_tiles;
                for (int k = w.k0; k < w.k1 && !failed; ++k, ++st) {
                    const int sq = st % kPSQ;
                    if (st >= kPSQ && !mbar_wait<kWaitSlackNs>(bar_q_free + 8 * sq, (uint32_t)((st / kPSQ - 1) & 1), status, 61)) { failed = true; break; }
                    mbar_expect_tx(bar_q + 8 * sq, (uint32_t)C::QSTAGE);
                    tma_load_2d(q0 + (uint32_t)(sq * C::QSTAGE), &p.tm_q, k * C::QROW, rt * kPRows + rank * 128, bar_q + 8 * sq);
                    previous_launch();                                        // the activations are the pre-pass's
                    for (int h = 0; h < 2; ++h) {
                        const int ks = 2 * st + h, sx = ks % C::SX, prev = ks - C::SX;
                        if (prev >= 0 && !mbar_wait<kWaitSleepNs>(bar_done + 8 * (prev % kPDone), (uint32_t)((prev / kPDone) & 1), status, 62)) { failed = true; break; }
                        if (rank == 0) mbar_expect_tx(bar_x + 8 * sx, x_tx);
                        tma_load_2d_pair(x0 + (uint32_t)(sx * C::XTILE), &p.tm_x, (2 * k + h) * 64, tt * p.bn + rank * (p.bn / 2), x_pair0 + 8 * sx);
                    }
                }
            }
            // nothing of this CTA is in flight when it ends
            for (int ks = 2 * st > kPDone ? 2 * st - kPDone : 0; ks < 2 * st && !failed; ++ks)
                if (!mbar_wait<kWaitSleepNs>(bar_done + 8 * (ks % kPDone), (uint32_t)((ks / kPDone) & 1), status, 63)) failed = true;
        }
        __syncwarp();
    } else if (warp == kPTmaA) {
        // ------------------------------------------------------------------ factor tiles (64 of the step's 128 columns) and B
        if (lane == 0) {
            const uint32_t a_pair0 = map_to_rank(bar_a, 0), b_pair0 = map_to_rank(bar_b, 0);
            tma_prefetch_desc(&p.tm_a);
            tma_prefetch_desc(&p.tm_b);
            if (!p.b_early) previous_launch();
            while (!failed && sched.next(w)) {
                const int rt = w.tile / p.tok_tiles;
                if (st > 0) previous_launch();
                // the scale MMAs of the piece before have read its B
                if (st > 0 && !mbar_wait<kWaitSleepNs>(bar_a_free + 8 * ((st - 1) % kPSA), (uint32_t)(((st - 1) / kPSA) & 1), status, 64)) { failed = true; break; }
                if (rank == 0) mbar_expect_tx(bar_b, 2u * C::BTILE);
                tma_load_2d_pair(b_tile, &p.tm_b, 0, rt * kPRows + rank * 128, b_pair0);
                for (int k = w.k0; k < w.k1; ++k, ++st) {
                    const int sa = st % kPSA;
                    if (st >= kPSA) previous_launch();
                    if (st >= kPSA && !mbar_wait<kWaitSlackNs>(bar_a_free + 8 * sa, (uint32_t)((st / kPSA - 1) & 1), status, 65)) { failed = true; break; }
                    if (rank == 0) mbar_expect_tx(bar_a + 8 * sa, (uint32_t)(2 * p.r_pad * 128));
                    tma_load_2d_pair(a0 + (uint32_t)(sa * C::ATILE), &p.tm_a, (2 * k + rank) * 64, 0, a_pair0 + 8 * sa);
                }
            }
            for (int k = st > kPSA ? st - kPSA : 0; k < st && !failed; ++k)
                if (!mbar_wait<kWaitSleepNs>(bar_a_free + 8 * (k % kPSA), (uint32_t)((k / kPSA) & 1), status, 66)) failed = true;
        }
        __syncwarp();
    } else if (warp == kPScale) {
        // ------------------------------------------------------------------ scale MMAs (the pair's even CTA)
        // S of a step goes into the one buffer as soon as the workers of both CTAs have taken S of the step before
        if (rank == 0) {
            constexpr uint32_t idesc = umma_idesc_f16(1, 0, 1, kPRows, 128);                 // bf16, B operand MN-major, N = 128
            const uint32_t desc_hi = (uint32_t)(umma_desc_sw128(0, 1024, 16) >> 32), lbo_lo = (uint32_t)umma_desc_sw128(0, 1024, 16);
            const uint32_t b_lo = lbo_lo | ((b_tile & 0x3FFFFu) >> 4), a_lo0 = lbo_lo | ((a0 & 0x3FFFFu) >> 4);
            const uint32_t tmem_u = warp_uniform(tmem_base), leader = elect_one();
            const int ranks16 = p.r_pad / 16;
            for (int piece = 0; !failed && sched.next(w); ++piece) {
                if (piece > 0 || !p.b_early) previous_launch();
                if (!mbar_wait_warp<kWaitSleepNs>(bar_b, (uint32_t)(piece & 1), status, 69)) { failed = true; break; }
                for (int k = w.k0; k < w.k1; ++k, ++st) {
                    const int sa = st % kPSA;
                    if (st >= kPW / 2) previous_launch();                  // the workers stop there, and with them the steps behind
                    if (!mbar_wait_warp2(bar_a + 8 * sa, (uint32_t)((st / kPSA) & 1), bar_s_free, (uint32_t)((st + 1) & 1), status, 67)) { failed = true; break; }
                    tc_fence_after_sync();
                    const uint32_t a_lo = a_lo0 + (uint32_t)(sa * (C::ATILE >> 4));
                    for (int c = 0; c < ranks16; ++c)
                        umma2_f16_ss(tmem_u + kPSCol, umma_desc_pack(b_lo + c * 2, desc_hi), umma_desc_pack(a_lo + c * 128, desc_hi), idesc, c > 0, leader);
                    umma2_commit(bar_s, leader);
                    umma2_commit(bar_a_free + 8 * sa, leader);
                }
            }
        }
    } else if (warp == kPIssuer) {
        // ------------------------------------------------------------------ main MMAs (the pair's even CTA)
        // The tensor cores take in no more than an MMA or two ahead: whatever this warp does between the MMAs of two k-steps beyond about
        // 128 cycles leaves them idle.  A barrier that has long completed costs it about 120 cycles, hence one look at both of a
        // k-step's and the scale MMAs in a warp of their own (six looks a step in one warp: 1790 cycles a step, 1250 so, of which the MMAs themselves take 1152).
        if (rank == 0) {
            const uint32_t idesc = umma_idesc_f16(0, 0, 0, kPRows, 0) | ((uint32_t)(p.bn >> 3) << 17);
            const uint32_t desc_hi = (uint32_t)(umma_desc_sw128(0, 1024, 16) >> 32);
            const uint32_t x_lo0 = (uint32_t)umma_desc_sw128(0, 1024, 16) | ((x0 & 0x3FFFFu) >> 4);
            const uint32_t tmem_u = warp_uniform(tmem_base), leader = elect_one();
            previous_launch();
            for (int piece = 0; !failed && sched.next(w); ++piece) {
                if (piece > 0 && !mbar_wait_warp<kWaitSleepNs>(bar_acc_free, (uint32_t)((piece - 1) & 1), status, 70)) { failed = true; break; }
                for (int k = w.k0; k < w.k1 && !failed; ++k, ++st) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int ks = 2 * st + h, sx = ks % C::SX, ws = ks % kPW;
                        if (!mbar_wait_warp2(bar_w + 8 * ws, (uint32_t)((ks / kPW) & 1), bar_x + 8 * sx, (uint32_t)((ks / C::SX) & 1), status, 71)) { failed = true; break; }
                        tc_fence_after_sync();
                        const uint32_t wslot = tmem_u + kPWCol + (uint32_t)(ws * 32), x_lo = x_lo0 + (uint32_t)((sx * C::XTILE) >> 4);
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            umma2_f16_ts(tmem_u, wslot + c * 8, umma_desc_pack(x_lo + c * 2, desc_hi), idesc, (k > w.k0 || h > 0 || c > 0) ? 1u : 0u, leader);
                        umma2_commit(bar_done + 8 * (ks % kPDone), leader);
                    }
                }
                if (!failed) umma2_commit(bar_acc, leader);
            }
        }
    } else {
        // ------------------------------------------------------------------ workers
        const int g = warp >> 3, q = warp & 3, ch = (warp >> 2) & 1, row = q * 32 + lane;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16), lut_lane = lut + 4u * (uint32_t)lane;
        const uint32_t s_free0 = map_to_rank(bar_s_free, 0), w0 = map_to_rank(bar_w, 0), acc_free0 = map_to_rank(bar_acc_free, 0);
        int piece = 0;
        while (!failed && sched.next(w)) {
            for (int k = w.k0; k < w.k1; ++k, ++st) {
                const int sq = st % kPSQ, ks = 2 * st + g, ws = ks % kPW;
                if (!p.b_early || 2 * st >= kPW) previous_launch();
                if (!mbar_wait_warp2<kWaitSleepNs>(bar_s, (uint32_t)(st & 1), bar_q + 8 * sq, (uint32_t)((st / kPSQ) & 1), status, 73)) { failed = true; break; }
                tc_fence_after_sync();
                uint32_t s[32];
                tmem_ld_32x32(lane_addr + kPSCol + (uint32_t)(g * 64 + ch * 32), s);
                tmem_wait_ld(s);
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_pair(s_free0);                  // S is in registers
                uint32_t out[16];
                dequant_chunk<BITS>(q0 + (uint32_t)(sq * C::QSTAGE + row * C::QROW), row, g * 2 + ch, lut_lane, s, out);
                // the ring slot is free once the main MMA of four k-steps ago has read it
                const int prev = ks - kPW;
                if (prev >= 0 && !mbar_wait_warp<kWaitSleepNs>(bar_done + 8 * (prev % kPDone), (uint32_t)((prev / kPDone) & 1), status, 75)) { failed = true; break; }
                tc_fence_after_sync();
                tmem_st_32x16(lane_addr + kPWCol + (uint32_t)(ws * 32 + ch * 16), out);
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive_pair(w0 + 8 * ws);
                    mbar_arrive(bar_q_free + 8 * sq);
                }
            }
            if (failed) break;
            // ---------------------------------------------------------------- epilogue: lane = row, columns = tokens
            previous_launch();
            if (!mbar_wait_warp<kWaitSleepNs>(bar_acc, (uint32_t)(piece & 1), status, 76)) { failed = true; break; }
            tc_fence_after_sync();
            const int rt = w.tile / p.tok_tiles, tt = w.tile - rt * p.tok_tiles;
            const int i = rt * kPRows + rank * 128 + row;
            const bool to_scratch = w.k0 > 0;
            // the pairs that hold the rest of this tile's steps: the ones behind this one, up to the tile's end
            const long long left = (long long)(p.tiles - p.whole) * p.steps, tile_end = (long long)(w.tile - p.whole + 1) * p.steps;
            int others = 0;
            if (w.k0 == 0 && w.k1 < p.steps) {
                for (int o = pair + 1; o < p.pairs && o * left / p.pairs < tile_end; ++o) {
                    others = o - pair;
                    if (!__all_sync(0xffffffffu, piece_ready(p.flags + 2 * o + rank, kPWorkers, status, (uint32_t)o, 77))) { failed = true; break; }
                }
            }
            if (failed) break;
            // 16 tokens at a time, dealt out to the four warps of a row quadrant.  bf16 rows of y that are 16-byte multiples go through shared
            // memory: two 16-byte stores a lane instead of sixteen of 2 bytes (14336 x 4096, 1024 tokens: 115 us -> 110).
            const bool wide = !p.y_f32 && (p.m & 7) == 0;
            const uint32_t stage = stage0 + (uint32_t)(warp * C::STAGE);
#pragma unroll 1
            for (int c0 = (warp >> 2) * 16; c0 < p.bn; c0 += 64) {
                uint32_t v[16];
                tmem_ld_32x16(lane_addr + (uint32_t)c0, v);
                tmem_wait_ld(v);
                if (to_scratch) {
                    float4 *part = reinterpret_cast<float4 *>(p.partial + ((size_t)(2 * pair + rank) * p.bn + c0) * 128) + row;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        __stcg(part + c * 128, make_float4(__uint_as_float(v[4 * c]), __uint_as_float(v[4 * c + 1]), __uint_as_float(v[4 * c + 2]), __uint_as_float(v[4 * c + 3])));
                    continue;
                }
                float sum[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) sum[c] = __uint_as_float(v[c]);
                // the other pieces, two at a time in flight, added in a fixed order: along k
                for (int o0 = pair + 1; o0 <= pair + others; o0 += 2) {
                    float4 pv[2][4];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int o = o0 + j;
                        const bool has = o <= pair + others;
                        const float4 *part = reinterpret_cast<const float4 *>(p.partial + ((size_t)(2 * (has ? o : pair) + rank) * p.bn + c0) * 128) + row;
#pragma unroll
                        for (int c = 0; c < 4; ++c) pv[j][c] = has ? __ldcg(part + c * 128) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            sum[4 * c] += pv[j][c].x;
                            sum[4 * c + 1] += pv[j][c].y;
                            sum[4 * c + 2] += pv[j][c].z;
                            sum[4 * c + 3] += pv[j][c].w;
                        }
                }
                const int tok0 = tt * p.bn + c0;
                if (wide) {
                    __syncwarp();                            // the lanes have read the tokens before
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        asm volatile("st.shared.u16 [%0], %1;" ::"r"(stage + (uint32_t)(c * 64 + lane * 2)), "h"(__bfloat16_as_ushort(__float2bfloat16_rn(sum[c]))) : "memory");
                    __syncwarp();
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int tok = tok0 + h * 8 + (lane >> 2), i8 = i - lane + (lane & 3) * 8;       // eight rows of one token
                        const uint4 o = lds_v4(stage + (uint32_t)((h * 32 + lane) * 16));
                        if (tok < p.M && i8 < p.m) *reinterpret_cast<uint4 *>(static_cast<uint16_t *>(p.y) + (size_t)tok * p.m + i8) = o;
                    }
                } else if (i < p.m) {
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        if (tok0 + c < p.M) store_out(p.y, p.y_f32, (size_t)(tok0 + c) * p.m + i, sum[c]);
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_pair(acc_free0);
            piece_done(p.flags, pair, rank, others, to_scratch, kPWorkers, lane);
            ++piece;
        }
    }

    if (failed) ptx::record_give_up(p.status, LORDS_ERR_TIMEOUT);
    tc_fence_before_sync();
    __syncthreads();
    // neither CTA leaves while the other may still signal its barriers or read its operands
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == kPTmaA) {
        tc_fence_after_sync();
        tmem_dealloc2(tmem_base, kPTmemCols);
    }
}

template <int BITS, int RP> struct PairVariant {
    static void fill(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int pairs, cudaStream_t stream)
    {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        // programmatic dependent launch: the kernel touches only weights until its griddepcontrol.wait
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg = cudaLaunchConfig_t{};
        cfg.gridDim = dim3((unsigned)(2 * pairs));
        cfg.blockDim = dim3(kPThreads);
        cfg.dynamicSmemBytes = PCfg<BITS, RP>::SMEM;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
    }
    // CTA pairs that can be resident at once
    static int resident(const State &st)
    {
        static int cache[kMaxDevices] = {};
        const int dev = device_slot(st);
        if (cache[dev] == 0) {
            if (cudaFuncSetAttribute(lords_umma_pair_kernel<BITS, RP>, cudaFuncAttributeMaxDynamicSharedMemorySize, PCfg<BITS, RP>::SMEM) != cudaSuccess) {
                (void)cudaGetLastError();
                return 0;
            }
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr[2];
            fill(cfg, attr, 1, nullptr);
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, lords_umma_pair_kernel<BITS, RP>, &cfg) != cudaSuccess) (void)cudaGetLastError();
            cache[dev] = n >= 1 ? n : -1;
        }
        return cache[dev] > 0 ? cache[dev] : 0;
    }
};

template <int BITS, int RP> int launch_pair_variant(const Problem &p, State &st, cudaStream_t stream)
{
    using V = PairVariant<BITS, RP>;
    const int pairs_max = V::resident(st);
    if (pairs_max < 1 || 2 * pairs_max > st.counter_slots) return LORDS_ERR_UNSUPPORTED;
    PairParams k;
    for (int c = 0; c < 16; ++c) k.levels[c] = p.levels[c];
    k.M = p.M; k.m = p.m;
    k.r_pad = (p.r + 15) / 16 * 16;
    k.steps = (p.n + 127) / 128;
    // token tiles as even as multiples of 32 allow
    k.tok_tiles = (p.M + kPTok - 1) / kPTok;
    k.bn = ((p.M + k.tok_tiles - 1) / k.tok_tiles + 31) / 32 * 32;
    const long long row_tiles = (p.m + kPRows - 1) / kPRows, tiles = row_tiles * k.tok_tiles;
    if (tiles > 0x3fffffffLL) return LORDS_ERR_UNSUPPORTED;
    k.tiles = (int)tiles;
    const Division division = divide_tiles(k.tiles, k.steps, pairs_max, 2, kMeetSteps);
    k.pairs = division.pairs;
    k.whole = division.whole;
    auto up = [](size_t b) { return (b + 1023) & ~(size_t)1023; };
    const int r8 = (p.r + 7) / 8 * 8;
    const bool pad_b = r8 != p.r;
    const size_t x_bytes = up((size_t)p.M * p.n * 2), b_bytes = pad_b ? up((size_t)p.m * r8 * 2) : 0;
    const size_t part_bytes = (size_t)k.pairs * 2 * k.bn * 128 * sizeof(float);
    if (x_bytes + b_bytes + part_bytes > st.workspace_bytes) return LORDS_ERR_WORKSPACE;
    void *const b_pad = pad_b ? st.workspace + x_bytes : nullptr;
    int rc = launch_umma_prepass(p, st.workspace, b_pad, stream);
    if (rc != LORDS_OK) return rc;
    k.b_early = !pad_b;
    k.partial = reinterpret_cast<float *>(st.workspace + x_bytes + b_bytes);
    k.flags = st.counters;
    k.y = p.y; k.y_f32 = p.y_f32;
    k.status = st.status_word;
    if (!make_map_2d(&k.tm_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, st.workspace, (uint64_t)p.n, (uint64_t)p.M, 64, (uint32_t)(k.bn / 2), CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&k.tm_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p.A, (uint64_t)p.n, (uint64_t)p.r, 64, (uint32_t)k.r_pad, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&k.tm_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, pad_b ? b_pad : static_cast<const void *>(p.B), (uint64_t)r8, (uint64_t)p.m, 64, 128,
                     CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&k.tm_q, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, p.q, (uint64_t)p.n * BITS / 8, (uint64_t)p.m, (uint32_t)PCfg<BITS, RP>::QROW, 128,
                     BITS == 4 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE))
        return LORDS_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    V::fill(cfg, attr, k.pairs, stream);
    LORDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, lords_umma_pair_kernel<BITS, RP>, k));
    st.last_launches = 2;
    st.last_path = "umma";
    return LORDS_OK;
}
template <int BITS> int launch_pair_bits(const Problem &p, State &st, cudaStream_t stream)
{
    return p.r <= 32 ? launch_pair_variant<BITS, 32>(p, st, stream) : launch_pair_variant<BITS, 64>(p, st, stream);
}

}  // namespace

int launch_umma_pair(const Problem &p, State &st, cudaStream_t stream)
{
    if (!umma_takes(p)) return LORDS_ERR_UNSUPPORTED;
    return p.bits == 4 ? launch_pair_bits<4>(p, st, stream) : p.bits == 3 ? launch_pair_bits<3>(p, st, stream) : launch_pair_bits<2>(p, st, stream);
}

}  // namespace lords
