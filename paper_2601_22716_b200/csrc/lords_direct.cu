// Direct path for few tokens: W^ = L[Q] (.) (BA) is formed in registers and multiplied there.
//
// A warp owns 16 rows of W^.  Per 32 columns it forms S = B A with warp-level MMAs (Eq. 3; bf16 operands, fp32 sums),
// multiplies them by the levels of the codes (lane-private table) and feeds the products straight to the next MMA as its
// left operand: the accumulator layout of one MMA is the operand layout of the other, so nothing of W^ leaves the
// register file, and there is no hand-over between warps but one barrier per 64-column strip.  Rows need no
// alignment and any rank goes.
//
// Two forms.  Layers that the 16-token and the scale-MMA kernel take as well have the operands of those kernels: S, the levels, W^ and x
// in fp16.  All others (EXACT: ragged rows, ranks above 64; and one or two tokens) hold S, the levels and W^ in fp32, as the CUDA-core
// path does: W^ enters the product as three bf16 parts, x as it is.  Tensor cores cut sums off instead of rounding
// them, so S of every 16 ranks and the first parts' products of every 16 columns start from zero and are added on the
// CUDA cores; the lower parts' products, 2^-8 of the sum, keep to the tensor cores.  Error of the fp32 sums
// against 64 bits, norms, normal activations, 256 x 256 to 1024 x 14336, ranks 4 to 128: 6e-8 to 1.7e-7 (CUDA cores 8e-8 to 1.6e-7; the
// fp16 form 2e-4 to 3.3e-4).  37 tokens of 1000 x 2730, rank 10: 12.7 us a call (CUDA cores 67.6).
//
// A cluster shares one tile of 128 rows and splits its columns; every CTA sends its partial sums to the CTA that owns
// the row (asynchronous stores counted on that CTA's barrier), which adds them in rank order: deterministic,
// no atomics, no trip through global memory.  Tokens that one CTA does not take are further groups of CTAs (grid y), each of which
// forms W^ again: EXACT takes up to 32 (with groups of 16 and ranks in steps of 32 before, 48 tokens: 4096 x 4094, rank 32, 64.0 us, 44.8 so;
// 5472 x 10524, rank 11, 170 and 119; 37 tokens of 1000 x 2730, rank 10, 15.0 and 12.7).
//
// Bound: warp instructions -- four per code pair for the table and the product (EXACT: some twenty), the MMAs (2 RK + M / 8, or
// 3 M / 8, per 16 x 16 weights at the warp-level rate) and the loads around them; codes, factors and activations come by
// asynchronous copies several strips ahead.  CTAs are small (eight warps, at most 111 KB), so that two or more share an SM
// and the next call's CTAs set up (and, where that call is not `late`, load their weights) while this call computes (programmatic
// dependent launch).
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

constexpr int kWarps = 8, kThreads = kWarps * 32;
constexpr int kRows = kWarps * 16;                  // rows of W^ per CTA
constexpr int kCols = 64;                           // columns per strip
constexpr int kClusterMax = 16;
constexpr int kTokenMax = 128;                      // beyond, the two-phase and the scale-MMA kernels, which form W^ less often
constexpr int kAPitch = kCols * 2 + 16;             // bytes per rank (or token) row: ldmatrix reads eight rows without bank conflicts
constexpr int kQPitch = 48;                         // bytes per code row: eight rows in eight different 16-byte bank groups

// BITS: code width.  RK: rank in steps of 16 (zero padded).  MT: tokens (8 to 32, zero padded).
template <int BITS, int RK, int MT, bool ALIGNED, bool EXACT> struct DirCfg {
    static constexpr int ENTRIES = 1 << 2 * BITS;                             // level pairs
    static constexpr int LUT = ENTRIES * 128;                                 // 32 lane-private copies of every pair (EXACT: 16 of 8 bytes)
    static constexpr int SA = RK <= 2 || (RK == 4 && MT < 24) ? 3 : 2;        // strips of A and x in flight
    // Strips of codes in flight.  Codes that are not ALIGNED wait in registers instead, and two stages do; the SM so keeps 56 KB of its
    // 256 as L1 beside two CTAs, not 23, which the words of x that are loaded by turns want (32 tokens, 5472 x 10524, rank 11: 88 us
    // with 23 KB, 74 with 56).
    static constexpr int SQ = ALIGNED ? 4 : 2;
    static constexpr int ASTAGE = RK * 16 * kAPitch;
    static constexpr int XPART = MT * kAPitch;
    static constexpr int XSTAGE = EXACT ? 2 * XPART : XPART;                  // EXACT: x, and x without infinities and NaNs
    static constexpr int QSTAGE = kRows * kQPitch;
    // Partial sums received: cluster x rows owned x tokens.  The owner's lanes read one token of 32 rows, which with the pairs of tokens in
    // order would meet in two to eight banks: pair u of a row sits at u ^ red_swizzle(row).  A remote store of four pairs keeps to
    // one 32-byte sector; rows padded by a pair instead, which stores then straddle, took 2 % longer with eight tokens (1344 x 704, rank 5:
    // 3.41 us, 3.20 so) and gained less with more (2880 x 1792, rank 9, 14 tokens: 7.7 us in order, 6.9 padded, 6.4 so).
    static constexpr int RED_SHIFT = MT == 32 ? 0 : MT == 16 ? 1 : 2, RED_MASK = MT == 32 ? 15 : MT == 16 ? 7 : 3;
    static __device__ __forceinline__ int red_swizzle(int row) { return row >> RED_SHIFT & RED_MASK; }
    static constexpr int RED = (kRows + kClusterMax) * MT * 4;
    static constexpr int SMEM = LUT + SA * ASTAGE + 2 * XSTAGE + SQ * QSTAGE + RED + 16;
};

struct DirectParams {
    const uint16_t *x;
    const uint8_t *q;
    const uint16_t *B;
    const uint16_t *A;
    float levels[16];
    int M, m, n, r;
    int strips;            // 64-column strips per row
    int late;              // nothing is read before the previous launch has ended (stream_ordered)
    int per_rank;          // rows of the tile that one CTA of the cluster adds up: ceil(128 / cluster)
    uint32_t per_rank_inv; // ceil(65536 / per_rank): row / per_rank by a multiplication
    void *y;
    int y_f32;
    int *status;
};

template <int BITS, int RK, int MT, bool ALIGNED, bool EXACT>
__global__ void __launch_bounds__(kThreads, EXACT || RK > 4 ? 2 : 3) lords_direct_kernel(const DirectParams p)
{
    using C = DirCfg<BITS, RK, MT, ALIGNED, EXACT>;
    constexpr int TG = MT / 8;                      // groups of eight tokens
    extern __shared__ __align__(1024) uint8_t dir_smem[];
    const uint32_t lut = smem_u32(dir_smem);
    const uint32_t a_s = lut + C::LUT, x_s = a_s + C::SA * C::ASTAGE, q_s = x_s + 2 * C::XSTAGE;
    const uint32_t red = q_s + C::SQ * C::QSTAGE, bar = red + C::RED;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;

    const int csize = (int)cluster_nctarank(), rank = (int)cluster_ctarank();
    const int row0 = ((int)blockIdx.x / csize) * kRows;
    const int s_a = rank * p.strips / csize, total = (rank + 1) * p.strips / csize - s_a;
    const size_t row_bytes = (size_t)p.n * BITS / 8;
    const uint8_t *q_end = p.q + (size_t)p.m * row_bytes;

    // rows of the tile that this CTA adds up in the end
    const int per_rank = p.per_rank;
    const int tok0 = (int)blockIdx.y * MT, ntok = p.M - tok0 < MT ? p.M - tok0 : MT;
    const int own0 = rank * per_rank, own_n = own0 >= kRows ? 0 : (own0 + per_rank < kRows ? per_rank : kRows - own0);
    if (csize > 1) {
        if (tid == 0) {
            mbar_init(bar, 1);
            fence_mbar_init();
            mbar_expect_tx(bar, (uint32_t)(csize * own_n * ((ntok + 1) / 2) * 8));    // every pair of tokens that exists
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // waited for before the first remote store
    }

    // ---- loads of one strip -------------------------------------------------------------------------------
    // codes: 8 * BITS bytes per row.  ALIGNED: asynchronous copies.  Otherwise (any byte alignment) aligned words are
    // loaded into registers one iteration ahead and put together by funnel shifts on their way to shared memory.
    constexpr int CB = BITS == 3 ? 8 : 16, CH = kCols * BITS / 8 / CB;       // chunk bytes, chunks per row (2, 3, 1)
    constexpr int QIT = (kRows * CH + kThreads - 1) / kThreads, QW = CB / 4;
    uint32_t qraw[ALIGNED ? 1 : QIT][QW + 1];
    auto chunk_of = [&](int it, int k, bool &in, int &row, int &ch) -> const uint8_t * {
        const int e = tid + k * kThreads;
        row = e / CH; ch = e % CH;
        const int i = row0 + row, byte = (s_a + it) * (kCols * BITS / 8) + ch * CB;
        in = row < kRows && i < p.m && byte < (int)row_bytes;
        return p.q + (in ? (size_t)i * row_bytes + byte : 0);
    };
    auto stage_q = [&](int it) {                     // ALIGNED
        if (it < total)
#pragma unroll
            for (int k = 0; k < QIT; ++k) {
                bool in; int row, ch;
                const uint8_t *src = chunk_of(it, k, in, row, ch);
                const uint32_t dst = q_s + (uint32_t)((it % C::SQ) * C::QSTAGE + row * kQPitch + ch * CB);
                if ((kRows * CH) % kThreads == 0 || row < kRows) {
                    if constexpr (CB == 16) cp_async16(dst, src, in ? 16 : 0);
                    else cp_async8(dst, src, in ? 8 : 0);
                }
            }
    };
    auto load_q = [&](int it) {                      // not ALIGNED
#pragma unroll
        for (int k = 0; k < QIT; ++k) {
            bool in; int row, ch;
            const uint8_t *src = chunk_of(it < total ? it : 0, k, in, row, ch);
            const uint32_t *w = reinterpret_cast<const uint32_t *>(reinterpret_cast<uintptr_t>(src) & ~(uintptr_t)3);
#pragma unroll
            for (int b = 0; b <= QW; ++b) {
                qraw[ALIGNED ? 0 : k][b] = 0u;
                if (in && it < total) {
                    if (reinterpret_cast<const uint8_t *>(w + b + 1) <= q_end) qraw[ALIGNED ? 0 : k][b] = __ldg(w + b);
                    else
                        for (int d = 0; d < 4; ++d)  // the last word of the buffer, if it is not a whole one
                            if (reinterpret_cast<const uint8_t *>(w + b) + d < q_end)
                                qraw[ALIGNED ? 0 : k][b] |= (uint32_t) __ldg(reinterpret_cast<const uint8_t *>(w + b) + d) << (8 * d);
                }
            }
        }
    };
    auto store_q = [&](int it) {                     // not ALIGNED
        if (it < total)
#pragma unroll
            for (int k = 0; k < QIT; ++k) {
                bool in; int row, ch;
                const int sh = 8 * (int)(reinterpret_cast<uintptr_t>(chunk_of(it, k, in, row, ch)) & 3);
                const uint32_t dst = q_s + (uint32_t)((it % C::SQ) * C::QSTAGE + row * kQPitch + ch * CB);
                if (row < kRows)
#pragma unroll
                    for (int b = 0; b < QW; ++b) sts_u32(dst + 4 * b, __funnelshift_r(qraw[ALIGNED ? 0 : k][b], qraw[ALIGNED ? 0 : k][b + 1], sh));
            }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    // factor strip A[:, strip]: rows of A are 16-byte multiples (ALIGNED) or at least 4-byte ones (n is even)
    auto stage_a = [&](int it) {
        if (it < total) {
            const uint32_t dst0 = a_s + (uint32_t)((it % C::SA) * C::ASTAGE);
            const int col0 = (s_a + it) * kCols;
            constexpr int CB = ALIGNED ? 16 : 4, CH = kCols * 2 / CB;
#pragma unroll
            for (int k = 0; k < (RK * 16 * CH + kThreads - 1) / kThreads; ++k) {
                const int e = tid + k * kThreads, rk = e / CH, ch = e % CH, col = col0 + ch * (CB / 2);
                const bool in = rk < p.r && col < p.n;
                const uint16_t *src = p.A + (in ? (size_t)rk * p.n + col : 0);
                const uint32_t dst = dst0 + (uint32_t)(rk * kAPitch + ch * CB);
                if ((RK * 16 * CH) % kThreads == 0 || rk < RK * 16) {
                    if constexpr (ALIGNED) cp_async16(dst, src, in ? 16 : 0);
                    else cp_async4(dst, src, in ? 4 : 0);
                }
            }
        }
    };
    // activations: eight columns of one token per thread, converted on the way (registers one strip ahead)
    constexpr int XT = MT * (kCols / 8);             // threads that take part (64 to 256)
    static_assert(XT <= kThreads && MT % 8 == 0, "one chunk of x per thread");
    const int xt = tid / (kCols / 8), xc = tid % (kCols / 8) * 8;
    auto load_x = [&](int it, uint32_t (&v)[4]) {
        v[0] = v[1] = v[2] = v[3] = 0u;
        if (it < total && tid < XT && xt < ntok) {
            const int col = (s_a + it) * kCols + xc;
            const uint32_t *src = reinterpret_cast<const uint32_t *>(p.x + (size_t)(tok0 + xt) * p.n + col);
            if (ALIGNED) {
                if (col < p.n) {
                    const uint4 w = *reinterpret_cast<const uint4 *>(src);
                    v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (col + 2 * k < p.n) v[k] = src[k];
            }
        }
    };
    auto store_x = [&](int it, const uint32_t (&v)[4]) {
        if (tid < XT) {
            const uint32_t dst = x_s + (uint32_t)((it & 1) * C::XSTAGE + xt * kAPitch + xc * 2);
            uint32_t o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if constexpr (EXACT) {
                    o[k] = finite_pair(v[k]);
                } else {
                    const __half2 h = __floats2half2_rn(__uint_as_float(v[k] << 16), __uint_as_float(v[k] & 0xFFFF0000u));
                    o[k] = *reinterpret_cast<const uint32_t *>(&h);
                }
            }
            if constexpr (EXACT) sts_v4(dst, make_uint4(v[0], v[1], v[2], v[3]));
            sts_v4(dst + (EXACT ? C::XPART : 0), make_uint4(o[0], o[1], o[2], o[3]));
        }
    };

    if constexpr (EXACT) {
        fill_pair_table<BITS, false>(lut, p.levels, tid);
        if (p.late) {
            griddep_launch_dependents();
            griddep_wait();
        }
    }

    // ---- weights first: where the call is not `late` they do not depend on the previous launch.  Copies are committed in the order
    // q0, a0, q1, a1, q2, then per strip a + 2 and q + 3 (or, with two stages of A, q + 3 and a + 2 at its end).
    constexpr int kPending = C::SA == 3 ? 3 : 2;     // youngest copies that strip `it` does not need
    // What goes through registers (codes that are not ALIGNED, x, the fragments of B) is requested before any of it is waited for: one
    // way to memory, not three in a row.
    uint32_t xv[4];
    if constexpr (ALIGNED) stage_q(0);
    else load_q(0);
    commit();
    if (EXACT && p.late) load_x(0, xv);
    stage_a(0); commit();
    if constexpr (ALIGNED) stage_q(1);
    commit();
    stage_a(1); commit();
    if constexpr (ALIGNED) stage_q(2);
    commit();
    if constexpr (!EXACT) fill_pair_table<BITS, true>(lut, p.levels, tid);
    // B fragments of the warp's rows
    const int i0 = row0 + warp * 16 + g, i1 = i0 + 8;
    uint32_t bf[RK][4];
#pragma unroll
    for (int k = 0; k < RK; ++k)
#pragma unroll
        for (int h = 0; h < 4; ++h) bf[k][h] = load_b_pair(p.B, (h & 1) ? i1 : i0, k * 16 + 2 * t + ((h & 2) ? 8 : 0), p.m, p.r);

    if (!(EXACT && p.late)) {
        griddep_launch_dependents();
        griddep_wait();                              // x may be the previous launch's output
        load_x(0, xv);
    }
    if constexpr (!ALIGNED) { store_q(0); load_q(1); }
    store_x(0, xv);
    load_x(1, xv);

    float acc[TG][4], low[EXACT ? TG : 1][4];        // low: the sums of the weights' lower parts
#pragma unroll
    for (int k = 0; k < TG; ++k) acc[k][0] = acc[k][1] = acc[k][2] = acc[k][3] = 0.0f;
#pragma unroll
    for (int k = 0; k < (EXACT ? TG : 1); ++k) low[k][0] = low[k][1] = low[k][2] = low[k][3] = 0.0f;
    const uint32_t lut_lane = lut + (EXACT ? 8u * (uint32_t)(lane & 15) : 4u * (uint32_t)lane);

    for (int it = 0; it < total; ++it) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
        __syncthreads();            // strip `it` is in shared memory; the buffers refilled below have been read by everyone
        if constexpr (C::SA == 3) { stage_a(it + 2); commit(); }
        if constexpr (ALIGNED) stage_q(it + 3);
        else { store_q(it + 1); load_q(it + 2); }
        commit();
        store_x(it + 1, xv);
        load_x(it + 2, xv);
        const uint32_t a_tile = a_s + (uint32_t)((it % C::SA) * C::ASTAGE), x_tile = x_s + (uint32_t)((it & 1) * C::XSTAGE);
        const uint32_t q_row = q_s + (uint32_t)((it % C::SQ) * C::QSTAGE + (warp * 16 + g) * kQPitch);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            // S of 16 rows x 16 columns (eight-column tiles 2 h and 2 h + 1 of the 32).  EXACT, which is short of registers, forms it as it is
            // used, the fp16 form for all 32 columns at once
            float s[EXACT ? 2 : 4][4];
            auto add_ranks = [&](int k, int h, float (&s0)[4], float (&s1)[4]) {      // 16 ranks from 16 k on
                uint32_t v[4];
                ldmatrix_x4_trans(a_tile + (uint32_t)((k * 16 + (lane & 15)) * kAPitch + c * 64 + (2 * h + (lane >> 4)) * 16), v);
                if (k == 0) {
                    mma_bf16_first(s0, bf[k], v[0], v[1]);
                    mma_bf16_first(s1, bf[k], v[2], v[3]);
                } else if constexpr (EXACT) {
                    add_mma_bf16(s0, bf[k], v[0], v[1]);
                    add_mma_bf16(s1, bf[k], v[2], v[3]);
                } else {
                    mma_bf16(s0, bf[k], v[0], v[1]);
                    mma_bf16(s1, bf[k], v[2], v[3]);
                }
            };
            if constexpr (!EXACT) {
                // ranks outermost: four chains of MMAs side by side
#pragma unroll
                for (int k = 0; k < RK; ++k)
#pragma unroll
                    for (int h = 0; h < 2; ++h) add_ranks(k, h, s[2 * h], s[2 * h + 1]);
            }
            CodeWords<BITS> w0, w1;
            w0.read(q_row + (uint32_t)(c * 4 * BITS));
            w1.read(q_row + (uint32_t)(8 * kQPitch + c * 4 * BITS));
            // x of 32 columns: token row lane & 7, 16-byte chunk lane >> 3.  EXACT, which is short of registers, takes it 16 columns at
            // a time: chunk lane >> 3 & 1, and of a pair of token groups group lane >> 4
            const uint32_t x_lane = x_tile + (uint32_t)((lane & 7) * kAPitch + c * 64 +
                                                        (EXACT ? (TG > 1 ? (lane >> 4) * 8 * kAPitch : 0) + ((lane >> 3) & 1) * 16 : (lane >> 3) * 16));
            uint32_t xb[EXACT ? 1 : TG][4];
            if constexpr (!EXACT) {
#pragma unroll
                for (int k = 0; k < TG; ++k) ldmatrix_x4(x_lane + (uint32_t)(k * 8 * kAPitch), xb[k]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if constexpr (EXACT) {
#pragma unroll
                    for (int k = 0; k < RK; ++k) add_ranks(k, h, s[0], s[1]);
                    auto scales = [&](int u, int e) { return f32x2(s[u][e], s[u][e + 1]); };
                    const uint64_t w[4] = {w0.weights(2 * h, t, lut_lane, scales(0, 0)), w1.weights(2 * h, t, lut_lane, scales(0, 2)),
                                           w0.weights(2 * h + 1, t, lut_lane, scales(1, 0)), w1.weights(2 * h + 1, t, lut_lane, scales(1, 2))};
                    uint32_t hi[4], mid[4], lo[4];
                    split_weights(w, hi, mid, lo);
#pragma unroll
                    for (int k0 = 0; k0 < TG; k0 += 2) {
                        const uint32_t x_pair = x_lane + (uint32_t)(k0 * 8 * kAPitch + h * 32);
                        uint32_t xa[4], xf[4];
                        if (k0 + 1 < TG) {
                            ldmatrix_x4(x_pair, xa);
                            ldmatrix_x4(x_pair + (uint32_t)C::XPART, xf);
                        } else {
                            uint32_t v[2];
                            ldmatrix_x2(x_pair, v);
                            xa[0] = v[0]; xa[1] = v[1];
                            ldmatrix_x2(x_pair + (uint32_t)C::XPART, v);
                            xf[0] = v[0]; xf[1] = v[1];
                        }
#pragma unroll
                        for (int k = k0; k < (k0 + 2 < TG ? k0 + 2 : TG); ++k) {
                            add_mma_bf16(acc[k], hi, xa[2 * (k - k0)], xa[2 * (k - k0) + 1]);
                            mma_bf16(low[k], mid, xf[2 * (k - k0)], xf[2 * (k - k0) + 1]);
                            mma_bf16(low[k], lo, xf[2 * (k - k0)], xf[2 * (k - k0) + 1]);
                        }
                    }
                } else {
                    uint32_t wa[4];
                    wa[0] = scaled_pair(lds_table(w0.address(2 * h, t, lut_lane)), s[2 * h][0], s[2 * h][1]);
                    wa[1] = scaled_pair(lds_table(w1.address(2 * h, t, lut_lane)), s[2 * h][2], s[2 * h][3]);
                    wa[2] = scaled_pair(lds_table(w0.address(2 * h + 1, t, lut_lane)), s[2 * h + 1][0], s[2 * h + 1][1]);
                    wa[3] = scaled_pair(lds_table(w1.address(2 * h + 1, t, lut_lane)), s[2 * h + 1][2], s[2 * h + 1][3]);
#pragma unroll
                    for (int k = 0; k < TG; ++k) mma_f16(acc[k], wa, xb[k][2 * h], xb[k][2 * h + 1]);
                }
            }
        }
        if constexpr (C::SA == 2) {
            __syncthreads();        // two strips of A: the one just read is refilled only now
            stage_a(it + 2);
            commit();
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if constexpr (EXACT) {
#pragma unroll
        for (int k = 0; k < TG; ++k) add_low(acc[k], low[k]);
    }

    // ---- partial sums: lane holds rows g, g + 8 of the warp's tile, tokens 2t, 2t + 1 of each group
    bool failed = false;
    if (csize == 1) {
#pragma unroll
        for (int k = 0; k < TG; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int tok = k * 8 + 2 * t + (e & 1), i = (e & 2) ? i1 : i0;
                if (tok < ntok && i < p.m) store_out(p.y, p.y_f32, (size_t)(tok0 + tok) * p.m + i, acc[k][e]);
            }
        return;
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = warp * 16 + g + 8 * h, owner = (int)(((uint32_t)row * p.per_rank_inv) >> 16);
        const int own_row = row - owner * per_rank, swz = C::red_swizzle(own_row);
        const uint32_t dst = map_to_rank(red + (uint32_t)((rank * per_rank + own_row) * MT * 4), (uint32_t)owner);
        const uint32_t dbar = map_to_rank(bar, (uint32_t)owner);
#pragma unroll
        for (int k = 0; k < TG; ++k)
            if (k * 8 + 2 * t < ntok) st_async_cluster_2f32(dst + (uint32_t)(((k * 4 + t) ^ swz) * 8), acc[k][2 * h], acc[k][2 * h + 1], dbar);
    }
    if (own_n > 0) {
        if (!mbar_wait_cluster(bar, 0, p.status, 61)) failed = true;
        else
            for (int e = warp, groups = (own_n + 31) / 32; e < ntok * groups; e += kWarps) {
                const int tok = e / groups, row = (e - tok * groups) * 32 + lane, i = row0 + own0 + row;
                if (row < own_n) {
                    const int word = ((tok >> 1) ^ C::red_swizzle(row)) * 2 + (tok & 1);
                    float sum = 0.0f;
                    for (int rr = 0; rr < csize; ++rr) sum += __uint_as_float(lds_u32(red + (uint32_t)(((rr * per_rank + row) * MT + word) * 4)));
                    if (i < p.m) store_out(p.y, p.y_f32, (size_t)(tok0 + tok) * p.m + i, sum);
                }
            }
    }
    if (failed) ptx::record_give_up(p.status, LORDS_ERR_TIMEOUT);
    // no CTA leaves while stores of its own may be on their way to another
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

template <int BITS, int RK, int MT, bool ALIGNED, bool EXACT> struct DirectVariant {
    using C = DirCfg<BITS, RK, MT, ALIGNED, EXACT>;
    static void fill(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int cs, int tiles, int groups, cudaStream_t stream)
    {
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg = cudaLaunchConfig_t{};
        cfg.gridDim = dim3((unsigned)(tiles * cs), (unsigned)groups);
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
            auto kernel = lords_direct_kernel<BITS, RK, MT, ALIGNED, EXACT>;
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr[2];
            fill(cfg, attr, cs, 1, 1, nullptr);
            int n = 0;
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM) != cudaSuccess ||
                cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess)
                (void)cudaGetLastError();
            cache[dev][cs] = n >= 1 ? n : -1;
        }
        return cache[dev][cs] > 0 ? cache[dev][cs] : 0;
    }
    // The cluster size for this call and an estimate of its time, in strips of sixteen tokens: waves of clusters times (strips of a CTA
    // x the weight of its tokens + a fixed part worth two and a half).  A strip takes about as long
    // with two CTAs on an SM as with one (one alone waits for its own loads and MMAs: 4096 x 4096 split 4
    // ways, one CTA per SM, 16.6 us; split 8 ways, two per SM, 10.0), so what fits at once counts as one wave.
    static double plan(const DirectParams &k, int tiles, int forced, int dev, int &cs)
    {
        const int lim = kClusterMax < k.strips ? kClusterMax : k.strips, groups = (k.M + MT - 1) / MT;
        double best = 1e30;
        cs = 0;
        if (forced > 0) {
            for (cs = forced < lim ? forced : lim; cs > 1 && max_clusters(dev, cs) == 0;) --cs;
            best = groups;
        } else {
            for (int c = 1; c <= lim; ++c) {
                const int res = max_clusters(dev, c);
                if (res == 0) continue;
                const double t = (double)((tiles * groups + res - 1) / res) * ((k.strips + c - 1) / c * kStripWeight + 2.5);
                if (t <= best) { best = t; cs = c; }
            }
        }
        if (cs < 1 || max_clusters(dev, cs) == 0) best = 1e30;
        return best;
    }
    // Forming W^ takes most of a strip; every further group of eight tokens adds its three MMAs and their operands (one group of CTAs, 16,
    // 24, 32 tokens: 4096 x 4094, rank 32, 22.9, 25.8, 28.5 us; 5472 x 10524, rank 11, 55, 64, 74; 5000 x 4128, rank 60, 35, 42, 47).
    static constexpr double kStripWeight = MT <= 16 ? 1.0 : 1.0 + 0.2 * (MT / 8 - 2);
    static int launch(DirectParams &k, int tiles, int cs, bool ordered, cudaStream_t stream)
    {
        k.per_rank = (kRows + cs - 1) / cs;
        k.per_rank_inv = (uint32_t)((65536 + k.per_rank - 1) / k.per_rank);
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[2];
        fill(cfg, attr, cs, tiles, (k.M + MT - 1) / MT, stream);
        if (ordered) attr[1].val.programmaticStreamSerializationAllowed = 0;
        LORDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, lords_direct_kernel<BITS, RK, MT, ALIGNED, EXACT>, k));
        return LORDS_OK;
    }
};

// The first of the token widths MT with the least estimate.
template <int BITS, int RK, bool ALIGNED, bool EXACT, int... MT>
int launch_planned(DirectParams &k, const Problem &p, State &st, cudaStream_t stream)
{
    const int dev = device_slot(st), tiles = (p.m + kRows - 1) / kRows;
    double best = 1e29;
    int at = -1, best_cs = 0, i = 0, cs = 0;
    auto consider = [&](double t) { if (t < best) { best = t; at = i; best_cs = cs; } ++i; };
    (consider(DirectVariant<BITS, RK, MT, ALIGNED, EXACT>::plan(k, tiles, st.forced_splitk, dev, cs)), ...);
    int rc = LORDS_ERR_UNSUPPORTED;
    i = 0;
    ((i++ == at ? (void)(rc = DirectVariant<BITS, RK, MT, ALIGNED, EXACT>::launch(k, tiles, best_cs, p.ordered, stream)) : (void)0), ...);
    return rc;
}

template <int BITS, int RK, bool ALIGNED, bool EXACT> int launch_tokens(DirectParams &k, const Problem &p, State &st, cudaStream_t stream)
{
    if (p.M <= 8) return launch_planned<BITS, RK, ALIGNED, EXACT, 8>(k, p, st, stream);
    // More tokens to a group form W^ fewer times (EXACT, up to 64 ranks: beyond, the registers hold B); the fp16 form takes small
    // layers, where CTAs are few.  Without groups of 24, 55 layers off the grid took 4 % longer on average (6897 x 834, rank 42, 44 tokens:
    // 26.9 us, 34.4 without), without those of 32 3 % (3670 x 6944, rank 6, 32 tokens: 37.4 us, 58.0 without).
    if constexpr (EXACT && RK <= 4)
        if (p.M > 16) return launch_planned<BITS, RK, ALIGNED, EXACT, 16, 24, 32>(k, p, st, stream);
    return launch_planned<BITS, RK, ALIGNED, EXACT, 16>(k, p, st, stream);
}

template <int BITS, int RK, bool EXACT> int launch_direct(DirectParams &k, const Problem &p, State &st, cudaStream_t stream)
{
    const size_t row_bytes = (size_t)p.n * BITS / 8;
    const bool aligned = row_bytes % (BITS == 3 ? 8 : 16) == 0 && p.n % 8 == 0;
    if constexpr (EXACT)
        if (!aligned) return launch_tokens<BITS, RK, false, true>(k, p, st, stream);
    // the fp16 form: n is a multiple of 64 (128 for 3 bits), so its rows are aligned
    return launch_tokens<BITS, RK, true, EXACT>(k, p, st, stream);
}
template <int BITS> int launch_direct(DirectParams &k, const Problem &p, State &st, cudaStream_t stream)
{
    // fp16 operands only where the kernel this one stands in for has them (decode16, umma): what else ran on the CUDA cores in fp32, or,
    // with one or two tokens, on the reassociated form, keeps that range and precision
    if (umma_takes(p) && !decode_takes(p)) return p.r <= 32 ? launch_direct<BITS, 2, false>(k, p, st, stream) : launch_direct<BITS, 4, false>(k, p, st, stream);
    return p.r <= 16 ? launch_direct<BITS, 1, true>(k, p, st, stream)
         : p.r <= 32 ? launch_direct<BITS, 2, true>(k, p, st, stream)
         : p.r <= 64 ? launch_direct<BITS, 4, true>(k, p, st, stream) : launch_direct<BITS, 8, true>(k, p, st, stream);
}

template <int BITS, int RK, int MT> double estimate(const Problem &p, const State &st)
{
    using V = DirectVariant<BITS, RK, MT, true, false>;
    const int dev = device_slot(st), tiles = (p.m + kRows - 1) / kRows;
    DirectParams k;
    k.M = p.M;
    k.strips = (p.n + kCols - 1) / kCols;
    int cs = 0;
    if (V::plan(k, tiles, 0, dev, cs) >= 1e30) return 1e30;
    const int clusters = tiles * ((p.M + MT - 1) / MT), resident = V::max_clusters(dev, cs), waves = (clusters + resident - 1) / resident;
    const double sms = st.sm_count, work = (double)clusters * k.strips / sms, chain = (double)waves * ((k.strips + cs - 1) / cs);
    const double load = (double)(clusters < resident ? clusters : resident) * cs / sms;
    const bool high = RK > 2;
    return 0.71 + 1.1 * waves + (high ? 0.61 : 0.41) * chain + ((high ? 0.46 : 0.34) + (MT > 8 ? 0.06 : 0.0)) * work + 0.68 * load +
           (MT > 8 ? 0.59 : 0.0) + (high && p.r % 2 != 0 ? 0.68 : 0.0);
}
template <int BITS> double estimate(const Problem &p, const State &st)
{
    if (p.M <= 8) return p.r <= 32 ? estimate<BITS, 2, 8>(p, st) : estimate<BITS, 4, 8>(p, st);
    return p.r <= 32 ? estimate<BITS, 2, 16>(p, st) : estimate<BITS, 4, 16>(p, st);
}

}  // namespace

// The fp16 form: waves, the strips of one CTA (a chain of waits), all strips over the SMs (their instructions), the CTAs on an SM (which the next
// launch's find taken), and the fragments of B, one value at a time for odd ranks.  A least-squares fit to 340 layers of 0.06 to 59 M weights at
// 3 to 128 tokens, back to back, off by 7.5 % on average.
double direct_us(const Problem &p, const State &st) { return p.bits == 4 ? estimate<4>(p, st) : p.bits == 3 ? estimate<3>(p, st) : estimate<2>(p, st); }

// Up to kTokenMax tokens, any other dimension.
int launch_direct(const Problem &p, State &st, cudaStream_t stream)
{
    if (p.M > kTokenMax) return LORDS_ERR_UNSUPPORTED;
    DirectParams k;
    k.x = p.x; k.q = p.q; k.B = p.B; k.A = p.A;
    for (int c = 0; c < 16; ++c) k.levels[c] = p.levels[c];
    k.M = p.M; k.m = p.m; k.n = p.n; k.r = p.r;
    k.strips = (p.n + kCols - 1) / kCols;
    k.late = stream_ordered(p);
    k.y = p.y; k.y_f32 = p.y_f32;
    k.status = st.status_word;
    const int rc = p.bits == 4 ? launch_direct<4>(k, p, st, stream) : p.bits == 3 ? launch_direct<3>(k, p, st, stream) : launch_direct<2>(k, p, st, stream);
    if (rc != LORDS_OK) return rc;
    st.last_launches = 1;
    st.last_path = "direct";
    return LORDS_OK;
}

}  // namespace lords
