// Two-phase path for any shape: W^ = L[Q] (.) (BA) is expanded once into scratch, then one dense product
// y = x W^T runs on the tensor cores.
//
// The layers that come here (ragged rows, ranks above 64) are computed in 32 bits, as on the CUDA cores: S, the levels and W^ are
// fp32, W^ enters the product as three bf16 parts, x as it is (see split_weights).
//
//   expand:  S = B A by warp-level MMAs (Eq. 3; bf16 operands, fp32 sums in registers, every 16 ranks from zero), the level of every
//            code from a table of fp32 pairs, their product cut into its parts, which are stored row-major, one after the
//            other, each padded to a multiple of 64 columns.  The same launch copies the activations to rows of that
//            pitch, and once more without infinities and NaNs, which is what the lower parts are multiplied by.  No tensor map
//            touches the caller's tensors, so rows need no alignment and any rank goes.
//   product: tcgen05 on CTA pairs (cta_group::2, 256 rows of W^ x BN tokens per pair), both operands by TMA, three MMAs where one
//            would do in 16 bits.  Tensor cores cut sums off instead of rounding them, so the first parts' products of every 64
//            columns start from zero in one accumulator and the epilogue adds them up in registers, while the MMAs of the lower
//            parts, whose sum is 2^-8 of the other, run in a second accumulator.  The tiles of whole waves run one per pair; the
//            k-steps of the tiles left over are dealt out evenly over all pairs, and the pieces of a tile meet in scratch in a
//            fixed order (no atomics on data).
//
// Error of the fp32 sums against 64 bits, norms, normal activations, 200 to 1024 tokens: 1.0e-7 to 1.9e-7 (CUDA cores 1.7e-7 to 3.8e-7,
// W^ and x rounded to fp16 3e-4).
//
// When it pays: W^ is formed once for all tokens, where the CUDA cores (the only other path for most of these shapes) need r + M
// multiply-adds a weight: 5952 x 7008, r = 11, 578 tokens: 9160 us there, 248 here (81 with W^ in fp16, a third of the MMAs
// and of the scratch).
//
// Every wait is bounded; on expiry the role records LORDS_ERR_TIMEOUT and leaves its loop.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "lords_internal.h"
#include "lords_pair.cuh"
#include "lords_ptx.cuh"
#include "lords_tc_common.cuh"
#include "lords_warp_mma.cuh"

namespace lords {

namespace {

using namespace ptx;

// ------------------------------------------------------------------------------------------------- expand
constexpr int kExWarps = 16;
constexpr int kExThreads = kExWarps * 32;
constexpr int kExRows = kExWarps * 16;              // rows per CTA: 16 per warp
constexpr int kExCols = 64;                         // columns per strip
constexpr int kExStages = 3;                        // strips of A in flight
constexpr int kExPitch = kExCols * 2 + 16;          // bytes per rank row of a strip: 16 extra keep ldmatrix free of bank conflicts

template <int BITS, int RK> struct ExCfg {
    static constexpr int ENTRIES = BITS == 4 ? 256 : BITS == 3 ? 64 : 16;     // level pairs
    static constexpr int LUT = ENTRIES * 128;                                 // 16 copies of every pair in fp32, one for a lane of each half warp
    static constexpr int STAGE = RK * 16 * kExPitch;
    static constexpr int SMEM = LUT + kExStages * STAGE;
};

struct ExpandParams {
    const uint8_t *q;      // first row of this chunk
    const uint8_t *q_end;  // end of the whole packed buffer
    const uint16_t *B;     // first row of this chunk
    const uint16_t *A;
    const uint16_t *x;
    uint16_t *w16;         // [rows][3][np]: the parts of W^
    uint16_t *x16;         // [M][2][np]: the activations, and without infinities and NaNs
    float levels[16];
    int rows, n, np, r, M;
    int strips, splits;    // strips of 64 columns; CTAs that share a row tile's strips
    int w_blocks;          // blocks below this index expand, the others convert activations
    int late;              // nothing is read before the previous launch has ended (stream_ordered)
};

// The 8 codes at column c of a row (8 * BITS bits, c a multiple of 8), low code first.  ALIGNED: the row starts on a
// 4-byte boundary; otherwise anywhere, and the last bytes of the buffer are read one by one.
template <int BITS, bool ALIGNED>
__device__ __forceinline__ uint32_t load_codes8(const uint8_t *row, int c, const uint8_t *end)
{
    const uint8_t *p = row + (size_t)c * BITS / 8;       // 8 codes are BITS whole bytes
    if constexpr (ALIGNED && BITS == 4) {
        return __ldg(reinterpret_cast<const uint32_t *>(p));
    } else if constexpr (ALIGNED && BITS == 2) {
        return __ldg(reinterpret_cast<const uint16_t *>(p));
    } else {
        const uintptr_t a = reinterpret_cast<uintptr_t>(p);
        const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~(uintptr_t)3);
        const int sh = 8 * (int)(a & 3);
        if (reinterpret_cast<const uint8_t *>(w + 2) <= end) {
            const uint32_t lo = __ldg(w), hi = sh + 8 * BITS > 32 ? __ldg(w + 1) : 0u;
            return __funnelshift_r(lo, hi, sh);
        }
        uint32_t v = 0;
#pragma unroll
        for (int b = 0; b < BITS; ++b)
            if (p + b < end) v |= (uint32_t)p[b] << (8 * b);
        return v;
    }
}

// Bound: the write stream to L2 / HBM (6 bytes a weight against bits / 8 read); up to rank 64 the
// MMAs (rank / 8 per 16 x 8 tile at the warp-level rate) and the four instructions per code pair stay below it.
// RK: the rank in steps of 16 that the B fragments hold (zero padded).
template <int BITS, int RK, bool ALIGNED>
__global__ void __launch_bounds__(kExThreads, RK <= 4 ? 2 : 1) lords_expand_kernel(const ExpandParams p)
{
    using C = ExCfg<BITS, RK>;
    extern __shared__ __align__(128) uint8_t ex_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if ((int)blockIdx.x >= p.w_blocks) {
        // activations: eight columns of one token per thread, zeros from column n on
        griddep_launch_dependents();
        griddep_wait();
        const int chunks = p.np / 8;
        const size_t e = (size_t)((int)blockIdx.x - p.w_blocks) * kExThreads + tid;
        if (e < (size_t)p.M * chunks) {
            const size_t t = e / chunks;
            const int c = (int)(e % chunks) * 8;
            uint32_t w[4] = {0u, 0u, 0u, 0u};
            if (c < p.n) {
                const uint32_t *src = reinterpret_cast<const uint32_t *>(p.x + t * p.n + c);       // n is even: 4-byte aligned
                if ((p.n & 7) == 0) {
                    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(src));
                    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (c + 2 * k < p.n) w[k] = __ldg(src + k);
                }
            }
            uint16_t *dst = p.x16 + 2 * t * p.np + c;
            *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4 *>(dst + p.np) = make_uint4(finite_pair(w[0]), finite_pair(w[1]), finite_pair(w[2]), finite_pair(w[3]));
        }
        return;
    }

    const uint32_t lut = smem_u32(ex_smem), a_s = lut + C::LUT;
    const int tile = (int)blockIdx.x / p.splits, split = (int)blockIdx.x % p.splits;
    const int s_a = (int)((long long)split * p.strips / p.splits), s_b = (int)((long long)(split + 1) * p.strips / p.splits);
    const int row0 = tile * kExRows + warp * 16;
    const int g = lane >> 2, t = lane & 3;
    const int i0 = row0 + g, i1 = row0 + g + 8;

    fill_pair_table<BITS, false>(lut, p.levels, tid);
    const uint32_t lut_lane = lut + 8u * (uint32_t)(lane & 15);
    if (p.late) {
        griddep_launch_dependents();
        griddep_wait();
    }

    // A strip: RK * 16 ranks x 64 columns by 4-byte asynchronous copies (rows of A are 4-byte aligned, n being even),
    // zeros past rank r and past column n.  A thread moves column pairs; the pair (4 tt + u) of each group of 32
    // columns goes to position (4 u + tt), which hands a lane of the MMA eight consecutive columns over four tiles.
    auto stage_a = [&](int strip, int st) {
        const uint32_t dst0 = a_s + (uint32_t)(st * C::STAGE);
#pragma unroll
        for (int e = tid; e < RK * 16 * 32; e += kExThreads) {
            const int k = e >> 5, pr = e & 31, col = strip * kExCols + 2 * pr;
            const int pos = (pr & 16) | ((pr & 3) << 2) | ((pr >> 2) & 3);
            const bool in = k < p.r && col < p.n;
            cp_async4(dst0 + (uint32_t)(k * kExPitch + pos * 4), p.A + (in ? (size_t)k * p.n + col : 0), in ? 4 : 0);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int k = 0; k < kExStages - 1; ++k) {
        if (s_a + k < s_b) stage_a(s_a + k, k);
        else asm volatile("cp.async.commit_group;" ::: "memory");
    }

    // B fragments of the warp's 16 rows, kept for every strip
    uint32_t bf[RK][4];
#pragma unroll
    for (int k = 0; k < RK; ++k)
#pragma unroll
        for (int h = 0; h < 4; ++h) bf[k][h] = load_b_pair(p.B, (h & 1) ? i1 : i0, k * 16 + 2 * t + ((h & 2) ? 8 : 0), p.rows, p.r);

    const size_t row_bytes = (size_t)p.n * BITS / 8;
    const uint8_t *q0 = p.q + (size_t)i0 * row_bytes, *q1 = p.q + (size_t)i1 * row_bytes;
    uint32_t cur[2][2], nxt[2][2];          // [32-column group][row]: the lane's eight codes
    auto load_q = [&](int strip, uint32_t (&v)[2][2]) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int col = strip * kExCols + c * 32 + 8 * t;
            v[c][0] = (i0 < p.rows && col < p.n) ? load_codes8<BITS, ALIGNED>(q0, col, p.q_end) : 0u;
            v[c][1] = (i1 < p.rows && col < p.n) ? load_codes8<BITS, ALIGNED>(q1, col, p.q_end) : 0u;
        }
    };
    if (s_a < s_b) load_q(s_a, cur);

    griddep_launch_dependents();
    griddep_wait();                         // the previous call may still be reading the scratch that is overwritten below

    for (int s = s_a; s < s_b; ++s) {
        const int it = s - s_a;
        asm volatile("cp.async.wait_group %0;" ::"n"(kExStages - 2) : "memory");
        __syncthreads();                    // the strip is in; the stage refilled below has been read by everyone
        if (s + kExStages - 1 < s_b) stage_a(s + kExStages - 1, (it + kExStages - 1) % kExStages);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        if (s + 1 < s_b) load_q(s + 1, nxt);
        const uint32_t a_tile = a_s + (uint32_t)((it % kExStages) * C::STAGE);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            float acc[4][4];
#pragma unroll
            for (int k = 0; k < RK; ++k)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    // matrices: ranks 0-7 | 8-15 of the step for tile 2h, then for tile 2h + 1
                    uint32_t v[4];
                    ldmatrix_x4_trans(a_tile + (uint32_t)((k * 16 + (lane & 15)) * kExPitch + c * 64 + (2 * h + (lane >> 4)) * 16), v);
                    if (k == 0) {
                        mma_bf16_first(acc[2 * h], bf[k], v[0], v[1]);
                        mma_bf16_first(acc[2 * h + 1], bf[k], v[2], v[3]);
                    } else {
                        add_mma_bf16(acc[2 * h], bf[k], v[0], v[1]);
                        add_mma_bf16(acc[2 * h + 1], bf[k], v[2], v[3]);
                    }
                }
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
                const uint32_t w = cur[c][rr];
                uint64_t v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    // pair u of the lane's eight columns, at bit 2 BITS u
                    constexpr uint32_t mask = (uint32_t)(C::ENTRIES - 1) << 7;
                    const int off = 2 * BITS * u;
                    const uint32_t sh = off >= 7 ? w >> (off - 7) : w << (7 - off);
                    v[u] = f32x2_mul(lds_table64(lut_lane + (sh & mask)), f32x2(acc[u][2 * rr], acc[u][2 * rr + 1]));
                }
                uint32_t hi[4], mid[4], lo[4];
                split_weights(v, hi, mid, lo);
                const int i = rr ? i1 : i0;
                if (i < p.rows) {
                    uint16_t *dst = p.w16 + 3 * (size_t)i * p.np + s * kExCols + c * 32 + 8 * t;
                    *reinterpret_cast<uint4 *>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<uint4 *>(dst + p.np) = make_uint4(mid[0], mid[1], mid[2], mid[3]);
                    *reinterpret_cast<uint4 *>(dst + 2 * p.np) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) { cur[c][0] = nxt[c][0]; cur[c][1] = nxt[c][1]; }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// ------------------------------------------------------------------------------------------------ product
constexpr int kGRows = 256;                         // rows of W^ per CTA pair
constexpr int kGK = 64;                             // columns per k-step
constexpr int kGEpiWarp0 = 4;                       // warps from 4 on: epilogue; 0: TMA, 1: MMA issuer, 2: TMEM
constexpr uint32_t kGTmemCols = 512;

template <int BN> struct GCfg {
    static constexpr int EPI = BN >= 256 ? 16 : 8;               // epilogue warps (a k-step's first parts have to be read while the MMAs of its lower parts run: 2816 x 3072, 1024 tokens, 95 us with eight, 84 with sixteen)
    static constexpr int THREADS = (kGEpiWarp0 + EPI) * 32;
    static constexpr int ATILE = 128 * 128;                      // this CTA's 128 rows, 64 columns of one part
    static constexpr int BTILE = (BN / 2) * 128;                 // this CTA's half of the tokens
    static constexpr int STAGE = ATILE + BTILE;
    static constexpr int STAGES = BN >= 256 ? 6 : BN >= 128 ? 8 : 10;
    static constexpr int SMEM = 1024 + STAGES * STAGE + 256;
    static constexpr uint32_t ACC = BN < 32 ? 32 : BN;           // columns of one accumulator: first parts, lower parts
};

struct alignas(64) GemmParams {
    CUtensorMap tm_w;     // bf16 [rows][3 np], box {64, 128}, 128-byte swizzle (rows past the end read as zero)
    CUtensorMap tm_x;     // bf16 [M][2 np], box {64, BN / 2}
    int M, rows;          // rows of this chunk
    int row0, ldy;        // first row of the chunk inside y, row length of y
    int tok_tiles, tiles, ksteps, np;
    int pairs;            // CTA pairs launched
    int whole;            // tiles [0, whole) run unsplit, one per pair and wave; the k-steps of the rest are dealt out evenly
    float *partial;       // [pair][2][BN][128]: a piece that does not begin its tile
    int *flags;           // [pair][2]: warps that have put their part of the piece into scratch; zero between calls
    void *y;
    int y_f32;
    int *status;
};

template <int BN>
__global__ void __launch_bounds__(GCfg<BN>::THREADS, 1) lords_dense_kernel(const __grid_constant__ GemmParams p)
{
    using C = GCfg<BN>;
    constexpr int STAGES = C::STAGES;
    extern __shared__ uint8_t g_smem[];
    const uint32_t base = (smem_u32(g_smem) + 1023u) & ~1023u;
    const uint32_t bars = base + STAGES * C::STAGE;
    const uint32_t bar_full = bars, bar_empty = bars + 8 * STAGES;
    const uint32_t bar_acc_full = bar_empty + 8 * STAGES, bar_acc_empty = bar_acc_full + 16;
    const uint32_t tmem_slot = bar_acc_empty + 16;
    static_assert(8 * (2 * STAGES + 4) + 4 <= 256, "barrier area");

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster_ctarank();
    // Pairs are numbered against the launch order: a pair waits only for pieces of pairs with a lower block index,
    // which the hardware has started before it.
    const int pair = p.pairs - 1 - (int)(blockIdx.x >> 1);
    const int *status = p.status;
    bool failed = false;

    if (warp == 0) {
        if (lane < 2 * STAGES) mbar_init(bars + 8 * lane, 1);
        if (lane >= 2 * STAGES && lane < 2 * STAGES + 2) mbar_init(bars + 8 * lane, 1);                        // accumulator full: one commit
        if (lane >= 2 * STAGES + 2 && lane < 2 * STAGES + 4) mbar_init(bars + 8 * lane, 2 * C::EPI);           // read by both CTAs' epilogue
        fence_mbar_init();
        if (lane == 0) { tma_prefetch_desc(&p.tm_w); tma_prefetch_desc(&p.tm_x); }
    } else if (warp == 2) {
        tmem_alloc2(tmem_slot, kGTmemCols);
    }
    tc_fence_before_sync();
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");       // both CTAs' barriers exist
    tc_fence_after_sync();
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));
    griddep_launch_dependents();
    griddep_wait();                                                           // W^ and the fp16 activations are the previous launch's

    Schedule sched(p.pairs, p.whole, p.tiles, p.ksteps, pair);
    Piece w;
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA: this CTA's rows and its half of the tokens
        if (lane == 0) {
            const uint32_t full0 = map_to_rank(bar_full, 0);
            int it = 0;
            while (!failed && sched.next(w)) {
                const int rt = w.tile / p.tok_tiles, tt = w.tile - rt * p.tok_tiles;
                for (int j = 3 * w.k0; j < 3 * w.k1; ++j, ++it) {              // part j % 3 of k-step j / 3
                    const int s = it % STAGES, k = j / 3, part = j - 3 * k;
                    if (it >= STAGES && !mbar_wait(bar_empty + 8 * s, (uint32_t)((it / STAGES - 1) & 1), status, 51)) { failed = true; break; }
                    if (rank == 0) mbar_expect_tx(bar_full + 8 * s, 2u * C::STAGE);
                    const uint32_t dst = base + (uint32_t)(s * C::STAGE);
                    tma_load_2d_pair(dst, &p.tm_w, part * p.np + k * kGK, rt * kGRows + rank * 128, full0 + 8 * s);
                    tma_load_2d_pair(dst + C::ATILE, &p.tm_x, (part > 0 ? p.np : 0) + k * kGK, tt * BN + rank * (BN / 2), full0 + 8 * s);
                }
            }
            // nothing of this CTA is in flight when it ends: the last round of stages has been read
            for (int k = it > STAGES ? it - STAGES : 0; k < it && !failed; ++k)
                if (!mbar_wait(bar_empty + 8 * (k % STAGES), (uint32_t)((k / STAGES) & 1), status, 52)) failed = true;
        }
        __syncwarp();
    } else if (warp == 1 && rank == 0) {
        // ------------------------------------------------------------------ MMA issuer (the pair's even CTA)
        constexpr uint32_t idesc = umma_idesc_f16(1, 0, 0, kGRows, BN);
        const uint32_t desc_hi = (uint32_t)(umma_desc_sw128(0, 1024, 16) >> 32);
        const uint32_t lo0 = (uint32_t)umma_desc_sw128(0, 1024, 16) | ((base & 0x3FFFFu) >> 4);
        const uint32_t tmem_u = warp_uniform(tmem_base), leader = elect_one();
        int it = 0, steps = 0, pieces = 0;
        while (!failed && sched.next(w)) {
            for (int k = w.k0; k < w.k1 && !failed; ++k, ++steps) {
                if (steps > 0 && !mbar_wait_cluster(bar_acc_empty, (uint32_t)((steps - 1) & 1), status, 53)) { failed = true; break; }
                for (int part = 0; part < 3; ++part, ++it) {
                    if (part == 1 && k == w.k0 && pieces > 0 && !mbar_wait_cluster(bar_acc_empty + 8, (uint32_t)((pieces - 1) & 1), status, 57)) { failed = true; break; }
                    const int s = it % STAGES;
                    if (!mbar_wait_cluster(bar_full + 8 * s, (uint32_t)((it / STAGES) & 1), status, 54)) { failed = true; break; }
                    tc_fence_after_sync();
                    const uint32_t a_lo = lo0 + (uint32_t)((s * C::STAGE) >> 4), b_lo = a_lo + (C::ATILE >> 4);
                    const uint32_t acc = tmem_u + (part > 0 ? C::ACC : 0u);
                    const bool onto = part == 2 || (part == 1 && k > w.k0);   // first parts start from zero every k-step, lower ones every piece
#pragma unroll
                    for (int kk = 0; kk < kGK / 16; ++kk)
                        umma2_f16_ss(acc, umma_desc_pack(a_lo + kk * 2, desc_hi), umma_desc_pack(b_lo + kk * 2, desc_hi), idesc,
                                     (onto || kk > 0) ? 1u : 0u, leader);
                    umma2_commit(bar_empty + 8 * s, leader);
                    if (part == 0) umma2_commit(bar_acc_full, leader);
                    if (part == 2 && k == w.k1 - 1) umma2_commit(bar_acc_full + 8, leader);
                    __syncwarp();
                }
            }
            ++pieces;
        }
    } else if (warp >= kGEpiWarp0) {
        // ------------------------------------------------------------------ epilogue: lane = row, columns = tokens
        const int q = warp & 3, ch = (warp - kGEpiWarp0) >> 2;                // row quadrant, share of the columns
        const int row = q * 32 + lane;
        constexpr int CW = BN / (C::EPI / 4);
        static_assert(CW % 16 == 0, "columns are read sixteen at a time");
        const uint32_t empty0 = map_to_rank(bar_acc_empty, 0);
        const uint32_t acc = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * CW);
        int steps = 0, pieces = 0;
        while (!failed && sched.next(w)) {
            float sum[CW];
#pragma unroll
            for (int c = 0; c < CW; ++c) sum[c] = 0.0f;
            for (int k = w.k0; k <= w.k1; ++k) {
                // the first parts of a k-step, and after the last one the lower parts of the piece
                const bool lower = k == w.k1;
                if (!__all_sync(0xffffffffu, mbar_wait_cluster(bar_acc_full + (lower ? 8 : 0), (uint32_t)((lower ? pieces : steps) & 1), status, 55))) { failed = true; break; }
                tc_fence_after_sync();
#pragma unroll
                for (int c0 = 0; c0 < CW; c0 += 16) {
                    uint32_t v[16];
                    tmem_ld_32x16(acc + (lower ? C::ACC : 0u) + (uint32_t)c0, v);
                    tmem_wait_ld(v);
#pragma unroll
                    for (int c = 0; c < 16; c += 2) {
                        float a = __uint_as_float(v[c]), b = __uint_as_float(v[c + 1]);
                        if (lower) { a = a == a ? a : 0.0f; b = b == b ? b : 0.0f; }          // as add_low
                        f32x2_split(f32x2_add(f32x2(sum[c0 + c], sum[c0 + c + 1]), f32x2(a, b)), sum[c0 + c], sum[c0 + c + 1]);
                    }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_pair(empty0 + (lower ? 8 : 0));
                if (!lower) ++steps;
            }
            ++pieces;
            if (failed) break;
            const int rt = w.tile / p.tok_tiles, tt = w.tile - rt * p.tok_tiles;
            const int i = rt * kGRows + rank * 128 + row;                     // row of the chunk
            const bool to_scratch = w.k0 > 0;
            // the pairs that hold the rest of this tile's k-steps: the ones behind this one, up to the tile's end
            int others = 0;
            if (w.k0 == 0 && w.k1 < p.ksteps) {
                const long long left = (long long)(p.tiles - p.whole) * p.ksteps, tile_end = (long long)(w.tile - p.whole + 1) * p.ksteps;
                for (int o = pair + 1; o < p.pairs && o * left / p.pairs < tile_end; ++o) {
                    others = o - pair;
                    if (!__all_sync(0xffffffffu, piece_ready(p.flags + 2 * o + rank, C::EPI, status, (uint32_t)o, 56))) { failed = true; break; }
                }
            }
            if (failed) break;
#pragma unroll
            for (int c0 = 0; c0 < CW; c0 += 16) {
                const int col = ch * CW + c0;
                if (to_scratch) {
                    float *part = p.partial + ((size_t)(2 * pair + rank) * BN + col) * 128 + row;
#pragma unroll
                    for (int c = 0; c < 16; ++c) __stcg(part + (size_t)c * 128, sum[c0 + c]);
                } else {
                    // the other pieces, added in a fixed order: along k
                    for (int o = pair + 1; o <= pair + others; ++o) {
                        const float *part = p.partial + ((size_t)(2 * o + rank) * BN + col) * 128 + row;
                        float pv[16];
#pragma unroll
                        for (int c = 0; c < 16; ++c) pv[c] = __ldcg(part + (size_t)c * 128);
#pragma unroll
                        for (int c = 0; c < 16; ++c) sum[c0 + c] += pv[c];
                    }
                    if (i < p.rows) {
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            const int tok = tt * BN + col + c;
                            if (tok < p.M) store_out(p.y, p.y_f32, (size_t)tok * p.ldy + p.row0 + i, sum[c0 + c]);
                        }
                    }
                }
            }
            piece_done(p.flags, pair, rank, others, to_scratch, C::EPI, lane);
        }
    }

    if (failed) ptx::record_give_up(p.status, LORDS_ERR_TIMEOUT);
    tc_fence_before_sync();
    __syncthreads();
    // neither CTA leaves while the other may still signal its barriers or read its operands
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 2) {
        tc_fence_after_sync();
        tmem_dealloc2(tmem_base, kGTmemCols);
    }
}

// --------------------------------------------------------------------------------------------------- launch
template <int BITS, int RK, bool ALIGNED> int launch_expand(const ExpandParams &k, int blocks, bool early, const State &st, cudaStream_t stream)
{
    static bool done[kMaxDevices] = {};
    const int dev = device_slot(st);
    if (!done[dev]) {
        LORDS_CUDA_TRY(cudaFuncSetAttribute(lords_expand_kernel<BITS, RK, ALIGNED>, cudaFuncAttributeMaxDynamicSharedMemorySize, ExCfg<BITS, RK>::SMEM));
        done[dev] = true;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kExThreads);
    cfg.dynamicSmemBytes = ExCfg<BITS, RK>::SMEM;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    LORDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, lords_expand_kernel<BITS, RK, ALIGNED>, k));
    return LORDS_OK;
}
template <int BITS, int RK> int launch_expand(const ExpandParams &k, int blocks, bool aligned, bool early, const State &st, cudaStream_t stream)
{
    return aligned ? launch_expand<BITS, RK, true>(k, blocks, early, st, stream) : launch_expand<BITS, RK, false>(k, blocks, early, st, stream);
}
template <int BITS> int launch_expand(const ExpandParams &k, int blocks, bool aligned, bool early, const State &st, cudaStream_t stream)
{
    return k.r <= 32 ? launch_expand<BITS, 2>(k, blocks, aligned, early, st, stream)
                     : k.r <= 64 ? launch_expand<BITS, 4>(k, blocks, aligned, early, st, stream) : launch_expand<BITS, 8>(k, blocks, aligned, early, st, stream);
}

template <int BN> struct DenseVariant {
    static void fill(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int pairs, cudaStream_t stream)
    {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg = cudaLaunchConfig_t{};
        cfg.gridDim = dim3((unsigned)(2 * pairs));
        cfg.blockDim = dim3(GCfg<BN>::THREADS);
        cfg.dynamicSmemBytes = GCfg<BN>::SMEM;
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
            if (cudaFuncSetAttribute(lords_dense_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, GCfg<BN>::SMEM) != cudaSuccess) return 0;
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr[2];
            fill(cfg, attr, 1, nullptr);
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, lords_dense_kernel<BN>, &cfg) != cudaSuccess) (void)cudaGetLastError();
            cache[dev] = n >= 1 ? n : -1;
        }
        return cache[dev] > 0 ? cache[dev] : 0;
    }
    static size_t partial_bytes(int pairs) { return (size_t)pairs * 2 * BN * 128 * sizeof(float); }
};

template <int BN> int launch_product(GemmParams &k, const void *w16, const void *x16, int np, int pairs_max, const State &st, cudaStream_t stream)
{
    k.tok_tiles = (k.M + BN - 1) / BN;
    k.tiles = ((k.rows + kGRows - 1) / kGRows) * k.tok_tiles;
    k.ksteps = np / kGK;
    k.np = np;
    // (a k-step, twelve MMAs, is one and a half steps of the pair kernel)
    const Division division = divide_tiles(k.tiles, k.ksteps, pairs_max, 4, kMeetSteps / 1.5);
    k.pairs = division.pairs;
    k.whole = division.whole;
    if (!make_map_2d(&k.tm_w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, w16, (uint64_t)np * 3, (uint64_t)k.rows, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&k.tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, x16, (uint64_t)np * 2, (uint64_t)k.M, 64, BN / 2, CU_TENSOR_MAP_SWIZZLE_128B))
        return LORDS_ERR_CUDA;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    DenseVariant<BN>::fill(cfg, attr, k.pairs, stream);
    LORDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, lords_dense_kernel<BN>, k));
    return LORDS_OK;
}

template <int BN> int run_dense(const Problem &p, State &st, cudaStream_t stream)
{
    const int pairs = DenseVariant<BN>::resident(st);
    if (pairs < 1 || 2 * pairs > st.counter_slots) return LORDS_ERR_UNSUPPORTED;
    const int np = (p.n + 63) / 64 * 64;
    auto up = [](size_t b) { return (b + 1023) & ~(size_t)1023; };
    const size_t x_bytes = up((size_t)p.M * np * 4), part_bytes = up(DenseVariant<BN>::partial_bytes(pairs));
    if (x_bytes + part_bytes >= st.workspace_bytes) return LORDS_ERR_WORKSPACE;
    // rows per chunk: what the rest of the workspace holds (all rows, usually)
    long long chunk = (long long)((st.workspace_bytes - x_bytes - part_bytes) / ((size_t)np * 6));
    if (chunk >= p.m) {
        chunk = p.m;
    } else {
        // chunks of about equal size: a small last one would leave most pairs idle (5952 x 7008, 578 tokens: 308 us, 255 with equal ones)
        chunk /= kGRows;
        if (chunk < 1) return LORDS_ERR_WORKSPACE;
        const long long row_tiles = (p.m + kGRows - 1) / kGRows, chunks = (row_tiles + chunk - 1) / chunk;
        chunk = (row_tiles + chunks - 1) / chunks * kGRows;
    }
    if (chunk < 1) return LORDS_ERR_WORKSPACE;

    ExpandParams e;
    e.A = p.A; e.x = p.x;
    e.x16 = reinterpret_cast<uint16_t *>(st.workspace);
    e.w16 = reinterpret_cast<uint16_t *>(st.workspace + x_bytes + part_bytes);
    for (int c = 0; c < 16; ++c) e.levels[c] = p.levels[c];
    e.n = p.n; e.np = np; e.r = p.r; e.M = p.M;
    e.late = stream_ordered(p);
    e.strips = np / kExCols;
    const size_t row_bytes = (size_t)p.n * p.bits / 8;
    e.q_end = p.q + (size_t)p.m * row_bytes;
    const bool aligned = row_bytes % 4 == 0;
    GemmParams k;
    k.M = p.M; k.ldy = p.m;
    k.partial = reinterpret_cast<float *>(st.workspace + x_bytes);
    k.flags = st.counters;
    k.y = p.y; k.y_f32 = p.y_f32;
    k.status = st.status_word;
    int launches = 0;
    for (long long r0 = 0; r0 < p.m; r0 += chunk) {
        e.rows = (int)(p.m - r0 < chunk ? p.m - r0 : chunk);
        e.q = p.q + (size_t)r0 * row_bytes;
        e.B = p.B + (size_t)r0 * p.r;
        const int row_tiles = (e.rows + kExRows - 1) / kExRows;
        // at most two CTAs per SM in all (what is resident at once: a few more would run alone in a second wave)
        e.splits = 2 * st.sm_count / row_tiles;
        if (e.splits > e.strips / 2) e.splits = e.strips / 2;
        if (e.splits < 1) e.splits = 1;
        e.w_blocks = row_tiles * e.splits;
        const long long x_blocks = r0 == 0 ? ((long long)p.M * (np / 8) + kExThreads - 1) / kExThreads : 0;
        if (e.w_blocks + x_blocks > 2147483647LL) return LORDS_ERR_UNSUPPORTED;
        const int blocks = (int)(e.w_blocks + x_blocks);
        const bool early = !p.ordered || r0 > 0;
        int rc = p.bits == 4 ? launch_expand<4>(e, blocks, aligned, early, st, stream)
                             : p.bits == 3 ? launch_expand<3>(e, blocks, aligned, early, st, stream) : launch_expand<2>(e, blocks, aligned, early, st, stream);
        if (rc != LORDS_OK) return rc;
        k.rows = e.rows; k.row0 = (int)r0;
        rc = launch_product<BN>(k, e.w16, e.x16, np, pairs, st, stream);
        if (rc != LORDS_OK) return rc;
        launches += 2;
    }
    st.last_launches = launches;
    st.last_path = "dense";
    return LORDS_OK;
}

}  // namespace

// Any shape; LORDS_ERR_WORKSPACE when the workspace cannot hold the activations and one row tile of W^.
int launch_dense(const Problem &p, State &st, cudaStream_t stream)
{
    if (p.M <= 32) return run_dense<32>(p, st, stream);
    if (p.M <= 64) return run_dense<64>(p, st, stream);
    // token tile: 256 runs closest to the tensor cores' rate; 128 where it saves the larger part of a last tile
    const long long t256 = (p.M + 255) / 256 * 256, t128 = (p.M + 127) / 128 * 128;
    if (t128 * 5 < t256 * 4) return run_dense<128>(p, st, stream);
    return run_dense<256>(p, st, stream);
}

}  // namespace lords
