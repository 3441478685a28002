// Backward of the layer y = x W^T, W^ = L[Q] (.) (B A), with the codes fixed: the gradients that
// multiplicative fine-tuning of B and A needs (Sec. 3.4; the chain rule through S = BA is the one of
// Eq. 5).  With g = dL/dy (M x m):
//
//     dx = g W^                                   (M x n)
//     dS = (g^T x) (.) L[Q]                       (m x n, never stored: built tile by tile)
//     dB = dS A^T   (m x r),     dA = B^T dS      (r x n)
//
// dx is the forward operator of the transposed layer: W^T = L[Q^T] (.) (A^T B^T), so with a transposed
// copy of the packed codes (made once: the codes are frozen) and the transposed factors it runs on the
// forward kernels as they are.  This file holds what that needs -- the transposition of packed codes
// and of the two factors -- and the kernels for dB and dA.
//
// The same kernels give the straight-through gradients of quantisation-aware training (Sec. 3.3, Eq. 4-5):
// the tile of g^T x is dL/dW^ = dL/dW itself, and the factor of dL/dS is L[Q] - W (/) S instead of L[Q],
// with S = B A rebuilt per tile (by a scale MMA on the tensor schedule where the rank allows it).
//
// dB and dA: a tile of dS is formed by the product g^T x over the tokens, multiplied by the levels of
// the tile's codes, and folded with the matching column slice of A (for dB) and row slice of B (for
// dA); bf16 inputs are widened exactly, sums are fp32.  Three schedules:
//   tiles: one CTA per 64 x 64 tile of W, everything on the CUDA cores; it writes the tile's contributions to dB and dA into the library's
//          workspace, and a second kernel adds the contributions of a row (or column) of tiles in tile
//          order.  g^T x is formed once, and the grid fills the machine.  Taken when the workspace
//          holds the contributions (4 r (m n / 64 + n m / 64) bytes).
//   walk:  one CTA per 64 rows (dB) or 64 columns (dA) walks over the other dimension and keeps its
//          sums in registers.  No scratch memory, g^T x formed once per gradient.
//   tensor: the first schedule with the tile product g^T x on the tensor cores (tcgen05, bf16 operands
//          straight from g and x by TMA, fp32 accumulator in TMEM) and only the level multiply and
//          the two folds (register-blocked, operands from shared memory as 16-byte words) on the CUDA
//          cores.  Taken when the row pitches suit TMA (m, n multiples of 8).
// Either way every output element is summed in a fixed order without atomics: runs are bit-identical.
// Bound of the CUDA-core schedules: fp32 ALU, m n M fused multiply-adds for the tile product (twice with the walk).
#include <cuda.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "lords_internal.h"
#include "lords_ptx.cuh"
#include "lords_tc_common.cuh"

namespace lords {

namespace {

using namespace ptx;

__device__ __forceinline__ float bf16f(uint16_t h) { return __uint_as_float((uint32_t)h << 16); }

// Code (i, j) of a packed row-major code matrix with `row_bytes` bytes per row.
__device__ __forceinline__ uint32_t read_code(const uint8_t *__restrict__ q, size_t row_bytes, int i, int j, int bits)
{
    const uint8_t *row = q + (size_t)i * row_bytes;
    const int bit = j * bits, byte = bit >> 3, sh = bit & 7;
    uint32_t v = row[byte];
    if (sh + bits > 8) v |= (uint32_t)row[byte + 1] << 8;
    return (v >> sh) & ((1u << bits) - 1u);
}

// ---- transposition of packed codes -----------------------------------------------------------------
// A block turns 64 rows x 128 columns around in shared memory, one byte per code: a thread unpacks 32 codes of a row from
// whole words, another packs 32 codes of a column into whole words (two of them fill a 32-byte sector of a row of
// Q^T).  Bound: about five instructions per code and one shared-memory byte load; 4096 x 4096, 4 bits: 78 us when every thread
// collected its column code by code from global memory, 10 us now; 14336 x 4096, 3 bits: 27 (46 with a store of one word per
// row at a time).
constexpr int kTrRows = 64, kTrCols = 128, kTrPitch = kTrCols + 4, kTrThreads = 256;

template <int BITS>
__global__ void __launch_bounds__(kTrThreads) lords_transpose_codes_kernel(const uint8_t *__restrict__ Q, uint8_t *__restrict__ Qt, int m, int n)
{
    __shared__ __align__(16) uint8_t tile[kTrRows][kTrPitch];
    __shared__ uint32_t stage[BITS == 4 ? 1 : kTrThreads * BITS];
    const int tid = threadIdx.x, i0 = (int)blockIdx.y * kTrRows, j0 = (int)blockIdx.x * kTrCols;
    const size_t row_bytes = (size_t)n * BITS / 8, trow_bytes = (size_t)m * BITS / 8;
    constexpr uint32_t mask = (1u << BITS) - 1u;
    {
        const int row = tid >> 2, seg = tid & 3, i = i0 + row, j = j0 + seg * 32;
        uint32_t w[BITS + 1];                               // 32 codes are BITS words
#pragma unroll
        for (int k = 0; k <= BITS; ++k) w[k] = 0u;
        if (i < m && j < n) {
            const uint8_t *src = Q + (size_t)i * row_bytes + (size_t)j * BITS / 8;
            const int bytes = n - j >= 32 ? 4 * BITS : (n - j) * BITS / 8;
            if (bytes == 4 * BITS && (row_bytes & 3) == 0) {
#pragma unroll
                for (int k = 0; k < BITS; ++k) w[k] = __ldg(reinterpret_cast<const uint32_t *>(src) + k);
            } else if (bytes == 4 * BITS) {
                load_words_anywhere<BITS>(src, Q + (size_t)m * row_bytes, w);
            } else {
#pragma unroll
                for (int k = 0; k < 4 * BITS; ++k)
                    if (k < bytes) w[k >> 2] |= (uint32_t)__ldg(src + k) << (8 * (k & 3));
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            uint32_t v = 0;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int bit = (4 * q + e) * BITS, wi = bit >> 5, sh = bit & 31;
                const uint32_t c = (sh + BITS > 32 ? __funnelshift_r(w[wi], w[wi + 1], sh) : w[wi] >> sh) & mask;
                v |= c << (8 * e);
            }
            *reinterpret_cast<uint32_t *>(&tile[row][seg * 32 + 4 * q]) = v;
        }
    }
    __syncthreads();
    {
        const int col = tid & (kTrCols - 1), half = tid >> 7, j = j0 + col, i = i0 + half * 32;
        if (j - (tid & 31) < n && i < m) {                  // per warp
            uint32_t w[BITS + 1];
#pragma unroll
            for (int k = 0; k <= BITS; ++k) w[k] = 0u;
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const uint32_t c = tile[half * 32 + e][col];
                const int bit = e * BITS, wi = bit >> 5, sh = bit & 31;
                w[wi] |= c << sh;
                if (sh + BITS > 32) w[wi + 1] |= c >> (32 - sh);
            }
            uint8_t *dst = Qt + (size_t)j * trow_bytes + (size_t)i * BITS / 8;
            const int bytes = m - i >= 32 ? 4 * BITS : (m - i) * BITS / 8;      // m is a multiple of the pack group
            if (bytes == 4 * BITS && (trow_bytes & 3) == 0) {
                if constexpr (BITS != 4) {
                    const int j0w = j - (tid & 31);
                    store_codes_staged<BITS>(ptx::smem_u32(stage) + (uint32_t)((tid >> 5) * 32 * BITS * 4), Qt + (size_t)j0w * trow_bytes + (size_t)i * BITS / 8,
                                             trow_bytes, n - j0w, tid & 31, w);
                } else if (j < n && (trow_bytes & 15) == 0) {
                    *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
                } else if (j < n) {
#pragma unroll
                    for (int k = 0; k < BITS; ++k) reinterpret_cast<uint32_t *>(dst)[k] = w[k];
                }
            } else if (j < n && bytes == 4 * BITS) {
                store_words_anywhere<BITS>(dst, w);
            } else if (j < n) {
#pragma unroll
                for (int k = 0; k < 4 * BITS; ++k)
                    if (k < bytes) dst[k] = (uint8_t)(w[k >> 2] >> (8 * (k & 3)));
            }
        }
    }
}

// Two transpositions in one launch (the factors A and B of a layer): blocks [0, tiles0) take the first matrix,
// the others the second.
__global__ void lords_transpose_bf16_pair_kernel(const uint16_t *__restrict__ src0, uint16_t *__restrict__ dst0, int rows0, int cols0,
                                                 const uint16_t *__restrict__ src1, uint16_t *__restrict__ dst1, int rows1, int cols1,
                                                 int tiles0)
{
    __shared__ uint16_t tile[32][33];
    // A dependent launch on both sides: the next one (the pre-pass over the activations) may begin when all before this one has ended.
    griddep_wait();
    griddep_launch_dependents();
    const bool first = (int)blockIdx.x < tiles0;
    const uint16_t *src = first ? src0 : src1;
    uint16_t *dst = first ? dst0 : dst1;
    const int rows = first ? rows0 : rows1, cols = first ? cols0 : cols1;
    const int t = first ? (int)blockIdx.x : (int)blockIdx.x - tiles0, tiles_x = (cols + 31) / 32;
    const int c0 = (t % tiles_x) * 32, r0 = (t / tiles_x) * 32;
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int rr = r0 + k, cc = c0 + threadIdx.x;
        tile[k][threadIdx.x] = (rr < rows && cc < cols) ? src[(size_t)rr * cols + cc] : (uint16_t)0;
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int cc = c0 + k, rr = r0 + threadIdx.x;
        if (cc < cols && rr < rows) dst[(size_t)cc * rows + rr] = tile[threadIdx.x][k];
    }
}

// ---- dB and dA -------------------------------------------------------------------------------------------
constexpr int kT = 64;          // tile edge (rows of W and columns of W per step)
constexpr int kTok = 16;        // tokens per shared-memory slice of the g^T x product
constexpr int kBwThreads = 256;
constexpr int kRMaxBw = 128;    // = LORDS_R_MAX

struct BwParams {
    const uint16_t *g;    // bf16 [M][m]
    const uint16_t *x;    // bf16 [M][n]
    const uint8_t *q;     // packed codes [m][n * bits / 8]
    const uint16_t *B;    // bf16 [m][r]
    const uint16_t *A;    // bf16 [r][n]
    float levels[16];
    int bits, M, m, n, r;
    float *dB;            // [m][r]
    float *dA;            // [r][n]
    // quantisation-aware training (Eq. 4-5), schedule "walk": the latent weight (null: fine-tuning with
    // the codes fixed) and where dL/dW goes (null: not asked for)
    const uint16_t *W;    // bf16 [m][n]
    float *dW;            // float [m][n]
};

// ROLE 0: dB for rows blockIdx.x * 64 ..; ROLE 1: dA for columns blockIdx.x * 64 ...
// With p.W set the factor of dL/dS is L[Q] - W (/) S (Eq. 5; S = B A rebuilt per tile in fp32, summed over
// the rank in ascending order; 0 where S is 0), and the launch with write_dW set also stores the tile of
// g^T x as dL/dW (Eq. 4).
template <int ROLE>
__global__ void __launch_bounds__(kBwThreads) lords_backward_factors_kernel(const BwParams p, const int write_dW)
{
    __shared__ __align__(16) float gs[kTok][kT];   // g[t][i0 + ..]
    __shared__ __align__(16) float xs[kTok][kT];   // x[t][j0 + ..]
    __shared__ float ds[kT][kT + 1];               // dS tile
    __shared__ uint16_t fs[kRMaxBw][kT + 2];       // ROLE 0: A[k][j0 + ..]; ROLE 1: B[i0 + ..][k] stored [k][i]
                                                   // (rows 33 words apart: neighbouring k fall into different banks)
    __shared__ float lv_s[16];                     // the level table (a per-thread index into the kernel parameters is replayed per distinct value)

    const int tid = threadIdx.x;
    if (tid < 16) lv_s[tid] = p.levels[tid];       // read after the first __syncthreads below
    const int ty = tid >> 4, tx = tid & 15;   // 16 x 16 threads, a 4 x 4 micro-tile each
    const int own0 = blockIdx.x * kT;         // first owned row (ROLE 0) or column (ROLE 1)
    const int walk_len = ROLE == 0 ? p.n : p.m;
    const size_t row_bytes = (size_t)p.n * p.bits / 8;

    // accumulators: output element e = tid + 256 * a of the owned [64][r] (ROLE 0: [i][k]) or [r][64]
    // (ROLE 1: [k][j]) block
    // (r rounded up to a multiple of 4, so that the block is a whole number of elements per thread)
    constexpr int kAccMax = kRMaxBw * kT / kBwThreads;     // 32
    float acc[kAccMax];
    const int r4 = (p.r + 3) & ~3;
    const int nacc4 = r4 * kT / kBwThreads;
#pragma unroll
    for (int a = 0; a < kAccMax; ++a) acc[a] = 0.0f;

    for (int w0 = 0; w0 < walk_len; w0 += kT) {
        const int i0 = ROLE == 0 ? own0 : w0, j0 = ROLE == 0 ? w0 : own0;
        // ---- tile of g^T x over all tokens
        float c[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) c[a][b] = 0.0f;
        for (int t0 = 0; t0 < p.M; t0 += kTok) {
            for (int e = tid; e < kTok * kT; e += kBwThreads) {
                const int t = t0 + e / kT, cidx = e % kT;
                gs[e / kT][cidx] = (t < p.M && i0 + cidx < p.m) ? bf16f(p.g[(size_t)t * p.m + i0 + cidx]) : 0.0f;
                xs[e / kT][cidx] = (t < p.M && j0 + cidx < p.n) ? bf16f(p.x[(size_t)t * p.n + j0 + cidx]) : 0.0f;
            }
            __syncthreads();
#pragma unroll
            for (int t = 0; t < kTok; ++t) {
                const float4 g4 = *reinterpret_cast<const float4 *>(&gs[t][ty * 4]);
                const float4 x4 = *reinterpret_cast<const float4 *>(&xs[t][tx * 4]);
                const float gv[4] = {g4.x, g4.y, g4.z, g4.w}, xv[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) c[a][b] = fmaf(gv[a], xv[b], c[a][b]);
            }
            __syncthreads();
        }
        // ---- QAT: the tile of S = B A, by the same outer-product steps with the rank in place of the tokens
        float sc[4][4];
        if (p.W) {
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) sc[a][b] = 0.0f;
            for (int k0 = 0; k0 < p.r; k0 += kTok) {
                for (int e = tid; e < kTok * kT; e += kBwThreads) {
                    const int k = k0 + e / kT, cidx = e % kT;
                    gs[e / kT][cidx] = (k < p.r && i0 + cidx < p.m) ? bf16f(p.B[(size_t)(i0 + cidx) * p.r + k]) : 0.0f;
                    xs[e / kT][cidx] = (k < p.r && j0 + cidx < p.n) ? bf16f(p.A[(size_t)k * p.n + j0 + cidx]) : 0.0f;
                }
                __syncthreads();
#pragma unroll
                for (int t = 0; t < kTok; ++t) {
                    const float4 b4 = *reinterpret_cast<const float4 *>(&gs[t][ty * 4]);
                    const float4 a4 = *reinterpret_cast<const float4 *>(&xs[t][tx * 4]);
                    const float bv[4] = {b4.x, b4.y, b4.z, b4.w}, av[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) sc[a][b] = fmaf(bv[a], av[b], sc[a][b]);
                }
                __syncthreads();
            }
        }
        // ---- dS = (g^T x) (.) L[Q]   (QAT: (.) (L[Q] - W (/) S))
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int i = i0 + ty * 4 + a, j = j0 + tx * 4 + b;
                float lv = 0.0f;
                if (i < p.m && j < p.n) {
                    lv = lv_s[read_code(p.q, row_bytes, i, j, p.bits)];
                    if (p.W) {
                        lv = sc[a][b] != 0.0f ? lv - bf16f(p.W[(size_t)i * p.n + j]) / sc[a][b] : 0.0f;
                        if (write_dW) p.dW[(size_t)i * p.n + j] = c[a][b];
                    }
                }
                ds[ty * 4 + a][tx * 4 + b] = c[a][b] * lv;
            }
        // ---- the factor slice that folds the tile: A[:, j0 ..] (ROLE 0) or B[i0 .., :] (ROLE 1), zero padded
        for (int e = tid; e < r4 * kT; e += kBwThreads) {
            const int k = e / kT, cidx = e % kT;
            uint16_t v = 0;
            if (k < p.r) {
                if (ROLE == 0) { if (j0 + cidx < p.n) v = p.A[(size_t)k * p.n + j0 + cidx]; }
                else { if (i0 + cidx < p.m) v = p.B[(size_t)(i0 + cidx) * p.r + k]; }
            }
            fs[k][cidx] = v;
        }
        __syncthreads();
        // ---- fold: ROLE 0: dB[i][k] += sum_j dS[i][j] A[k][j];  ROLE 1: dA[k][j] += sum_i B[i][k] dS[i][j]
#pragma unroll
        for (int a = 0; a < kAccMax; ++a) {
            if (a >= nacc4) break;
            const int e = tid + kBwThreads * a;
            float s = acc[a];
            if (ROLE == 0) {
                const int i = e / r4, k = e % r4;
#pragma unroll 8
                for (int j = 0; j < kT; ++j) s = fmaf(ds[i][j], bf16f(fs[k][j]), s);
            } else {
                const int k = e / kT, j = e % kT;
#pragma unroll 8
                for (int i = 0; i < kT; ++i) s = fmaf(bf16f(fs[k][i]), ds[i][j], s);
            }
            acc[a] = s;
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < kAccMax; ++a) {
        if (a >= nacc4) break;
        const int e = tid + kBwThreads * a;
        if (ROLE == 0) {
            const int i = own0 + e / r4, k = e % r4;
            if (p.dB && i < p.m && k < p.r) p.dB[(size_t)i * p.r + k] = acc[a];
        } else {
            const int k = e / kT, j = own0 + e % kT;
            if (p.dA && k < p.r && j < p.n) p.dA[(size_t)k * p.n + j] = acc[a];
        }
    }
}

// Schedule "tiles": CTA (jt, it) handles rows it * 64 .. and columns jt * 64 .. of W.
//   part_dB[jt][i][k4]  (k4 < r4: r rounded up to a multiple of 4) and part_dA[it][k4][j]
__global__ void __launch_bounds__(kBwThreads) lords_backward_tile_kernel(const BwParams p, float *__restrict__ part_dB,
                                                                         float *__restrict__ part_dA)
{
    __shared__ __align__(16) float gs[kTok][kT];
    __shared__ __align__(16) float xs[kTok][kT];
    __shared__ float ds[kT][kT + 1];
    __shared__ uint16_t fs[kRMaxBw][kT + 2];
    __shared__ float lv_s[16];

    const int tid = threadIdx.x;
    if (tid < 16) lv_s[tid] = p.levels[tid];       // read after the first __syncthreads below
    const int ty = tid >> 4, tx = tid & 15;
    const int jt = blockIdx.x, it = blockIdx.y;
    const int i0 = it * kT, j0 = jt * kT;
    const size_t row_bytes = (size_t)p.n * p.bits / 8;
    const int r4 = (p.r + 3) & ~3;
    const int nacc4 = r4 * kT / kBwThreads;

    float c[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) c[a][b] = 0.0f;
    for (int t0 = 0; t0 < p.M; t0 += kTok) {
        for (int e = tid; e < kTok * kT; e += kBwThreads) {
            const int t = t0 + e / kT, cidx = e % kT;
            gs[e / kT][cidx] = (t < p.M && i0 + cidx < p.m) ? bf16f(p.g[(size_t)t * p.m + i0 + cidx]) : 0.0f;
            xs[e / kT][cidx] = (t < p.M && j0 + cidx < p.n) ? bf16f(p.x[(size_t)t * p.n + j0 + cidx]) : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < kTok; ++t) {
            const float4 g4 = *reinterpret_cast<const float4 *>(&gs[t][ty * 4]);
            const float4 x4 = *reinterpret_cast<const float4 *>(&xs[t][tx * 4]);
            const float gv[4] = {g4.x, g4.y, g4.z, g4.w}, xv[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) c[a][b] = fmaf(gv[a], xv[b], c[a][b]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = i0 + ty * 4 + a, j = j0 + tx * 4 + b;
            float lv = 0.0f;
            if (i < p.m && j < p.n) lv = lv_s[read_code(p.q, row_bytes, i, j, p.bits)];
            ds[ty * 4 + a][tx * 4 + b] = c[a][b] * lv;
        }
    if (part_dB) {
        for (int e = tid; e < r4 * kT; e += kBwThreads) {           // A[k][j0 ..], zero padded
            const int k = e / kT, cidx = e % kT;
            fs[k][cidx] = (k < p.r && j0 + cidx < p.n) ? p.A[(size_t)k * p.n + j0 + cidx] : (uint16_t)0;
        }
        __syncthreads();
        float *out = part_dB + ((size_t)jt * p.m + i0) * r4;
        for (int a = 0; a < nacc4; ++a) {
            const int e = tid + kBwThreads * a, i = e / r4, k = e % r4;
            float s = 0.0f;
#pragma unroll 8
            for (int j = 0; j < kT; ++j) s = fmaf(ds[i][j], bf16f(fs[k][j]), s);
            if (i0 + i < p.m) out[(size_t)i * r4 + k] = s;
        }
    }
    __syncthreads();
    if (part_dA) {
        for (int e = tid; e < r4 * kT; e += kBwThreads) {           // B[i0 ..][k] stored [k][i], zero padded
            const int k = e / kT, cidx = e % kT;
            fs[k][cidx] = (k < p.r && i0 + cidx < p.m) ? p.B[(size_t)(i0 + cidx) * p.r + k] : (uint16_t)0;
        }
        __syncthreads();
        float *out = part_dA + (size_t)it * r4 * p.n + j0;
        for (int a = 0; a < nacc4; ++a) {
            const int e = tid + kBwThreads * a, k = e / kT, j = e % kT;
            float s = 0.0f;
#pragma unroll 8
            for (int i = 0; i < kT; ++i) s = fmaf(bf16f(fs[k][i]), ds[i][j], s);
            if (j0 + j < p.n) out[(size_t)k * p.n + j] = s;
        }
    }
}

// Schedule "tensor": both products on the tensor cores.  A CTA takes a run of 128 x 128 tiles of W, row block after row block.  Per
// tile:
//   G[128 x 128] = sum_t g[t][i] x[t][j]   operands as they lie in memory (MN-major: a shared-memory row is one token), 64 tokens
//                                          per stage, accumulators in TMEM (two of them: the next tile's product
//                                          runs while this one is worked on)
//   dS = G (.) L[Q]                        sixteen epilogue warps, fp32
//   dB[128 x r] += dS A_tile^T,  dA_tile^T[128 x r] = dS^T B_tile
// The folds take dS as three bf16 terms, dS = hi + mid + lo exactly (8 bits of the significand each, split by truncation),
// and the factors are bf16 as given, so every product is exact.  Tensor cores cut their sums off instead of rounding them, about 1.5e-8 of
// the sum an MMA, which adds up where a sum goes through many: so a tile's product leaves TMEM in two sums over half of the tokens
// each (RAGGED, whose layers ran on the CUDA cores before: 32 or 64 tokens), a fold starts from zero with every tile, its smallest term
// first, and all these are added up rounding to nearest.  Error of dB and dA against 64 bits, norms: 3.3e-7 at 512 tokens (5.0e-7 with
// the folds on the CUDA cores and one sum over the tokens, 1.2e-6 with all sums in TMEM), RAGGED 1.6e-7 to 2.2e-7 (CUDA cores 2.0e-7 to
// 3.1e-7; 0.9e-6 to 3.4e-6); of dW at 1024 tokens 4.7e-7 (9.9e-7), RAGGED 1.0e-7 (2.5e-7; 1.0e-6).
// One shared-memory tile serves both folds, K-major for dB and MN-major (transposed) for dA; likewise the A tile and the B
// tile.  A CTA adds its tiles' contributions to dB of a row block in scratch; dA_tile goes there as one contribution per row block.
// 4096 x 4096, r = 32: 512 tokens 111 us with the folds on the CUDA cores (bound by shared memory at two multiply-adds per word
// read), 46 now (43 with the long sums in TMEM); QAT (with 67 MB of dW) 165 -> 74 (70), at 1024 tokens 81 (78); 4096 x 4094 at 1024
// tokens: factors 1361 -> 101 (76), QAT 16253 -> 184 (136).  What bounds it: with many tokens the way of g and x
// from L2 into shared memory (32 KB per 64 tokens of a tile, about 50 bytes a clock and SM), with few the epilogue (7 thousand cycles a
// tile; QAT 14, of which 5 for dW's stores and 3 for the quotients) and the first tile, which nothing overlaps.
//
// Warps 0..15: epilogue (eight of them: 47 and 94 us); 16: TMA of g and x; 17: main MMAs; 18: fold (and scale) MMAs; 19: TMA of the factor
// tiles.
constexpr int kTcRows = 128, kTcCols = 128, kTcTok = 64;
constexpr int kTcEpiWarps = 16;
constexpr int kTcTmaWarp = 16, kTcMainWarp = 17, kTcFoldWarp = 18, kTcFactorWarp = 19;
constexpr int kTcThreads = 20 * 32;
constexpr int kTcGAtom = kTcTok * 128;                        // 64 tokens x 64 rows (or columns) of W, bf16
constexpr int kTcStage = 4 * kTcGAtom;                        // g: two atoms, x: two
constexpr int kTcDsAtom = kTcRows * 128;                      // 128 rows x 64 columns of one term of dS
constexpr int kTcDsTerm = 2 * kTcDsAtom;

// RA: ranks the factor tiles are sized for (64 or 128).  QAT: with the scale tile and the latent weight (Eq. 4-5).
template <int RA, bool QAT> struct BwCfg {
    static constexpr int NA = QAT && RA == 64 ? 2 : 1;        // A tiles in flight: S of the next tile needs its A tile early
    static constexpr int STAGES = RA == 64 && !QAT ? 3 : 2;
    static constexpr int NG = QAT && RA == 128 ? 1 : 2;       // accumulators of G
    static constexpr int AATOM = RA * 128;                    // RA ranks x 64 columns
    static constexpr int ATILE = 2 * AATOM;
    static constexpr int BTILE = RA / 64 * kTcRows * 128;     // 128 rows x RA ranks, 64 ranks per atom
    static constexpr int WSTAGE = QAT && RA == 64 ? kTcEpiWarps * 1024 : 0;       // dW on its way out (with RA = 128 there is no room for it)
    static constexpr int SMEM = 1024 + STAGES * kTcStage + 3 * kTcDsTerm + NA * ATILE + BTILE + WSTAGE + 512;
    static constexpr uint32_t S_COL = NG * kTcCols, DB_COL = S_COL + (QAT ? kTcCols : 0);       // behind it dB and dA of one tile, or of two by turns
    static constexpr uint32_t TMEM = 512;
    static_assert(SMEM <= 232448 && DB_COL + 2 * RA <= 512, "shared memory and TMEM");
};

// Four fp32 sums in global memory, 16-byte aligned, each rounded to nearest.
__device__ __forceinline__ void red_add_v4(float *at, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(at), "f"(__uint_as_float(a)), "f"(__uint_as_float(b)), "f"(__uint_as_float(c)),
                 "f"(__uint_as_float(d)) : "memory");
}

// The division of all 128 x 128 tiles, row block after row block, into one run per CTA.  row_splits 0: equal runs, which may cross from a row
// block into the next (no CTA idles: 1024 tiles over 148 SMs are 7 rounds, four CTAs per row block 8); else that many runs per row
// block (the element-wise B tile is built once per CTA).
struct Runs {
    int row_blocks, col_tiles, ctas, row_splits;
    __host__ __device__ long long begin(int c) const
    {
        if (row_splits == 0) return (long long)row_blocks * col_tiles * c / ctas;
        return (long long)(c / row_splits) * col_tiles + (long long)col_tiles * (c % row_splits) / row_splits;
    }
    // the CTA whose run holds tile t
    __host__ __device__ int owner(long long t) const
    {
        const long long all = (long long)row_blocks * col_tiles;
        return (int)(((t + 1) * ctas + all - 1) / all - 1);
    }
    __host__ __device__ int first(int rb) const { return row_splits == 0 ? owner((long long)rb * col_tiles) : rb * row_splits; }
    __host__ __device__ int parts(int rb) const { return row_splits == 0 ? owner((long long)(rb + 1) * col_tiles - 1) - first(rb) + 1 : row_splits; }
};

struct alignas(64) BwTcParams {
    CUtensorMap tm_g;     // bf16 [M][m], box {64, 64}, 128-byte swizzle (tokens past M and rows past m read as zero)
    CUtensorMap tm_x;     // bf16 [M][n], box {64, 64}, 128-byte swizzle
    CUtensorMap tm_a;     // bf16 [r][n], box {64 columns, ceil16(r) ranks}, 128-byte swizzle (ranks past r read as zero)
    CUtensorMap tm_b;     // bf16 [m][r], box {64 ranks, 128 rows}, 128-byte swizzle; used if rows of B are 16-byte multiples
    BwParams b;
    int r4, r_pad;
    Runs runs;            // which tiles a CTA takes
    int fold_bufs;        // TMEM has room for dB and dA of one tile or of two
    int group;            // MMAs (of 16 tokens) of a tile's product whose sum is taken out of TMEM: 2, 4 or a multiple of 4
    float *part_dB;       // [contribution][m][r4] or null
    float *part_dA;       // [row blocks][r4][n] or null
    int *status;
};

// RAGGED: g, x or A are padded copies, and rows of W, dW and the codes may begin anywhere (checks that would cost the others 5 %).
template <int RA, bool QAT, bool RAGGED>
__global__ void __launch_bounds__(kTcThreads, 1) lords_backward_tc_kernel(const __grid_constant__ BwTcParams p)
{
    using C = BwCfg<RA, QAT>;
    extern __shared__ uint8_t tc_smem_raw[];
    const uint32_t base = (smem_u32(tc_smem_raw) + 1023u) & ~1023u;
    const uint32_t ds0 = base + C::STAGES * kTcStage, a_s = ds0 + 3 * kTcDsTerm, b_s = a_s + C::NA * C::ATILE, w_stage = b_s + C::BTILE, bars = w_stage + C::WSTAGE;
    const uint32_t bar_full = bars, bar_empty = bar_full + 8 * C::STAGES, bar_g = bar_empty + 8 * C::STAGES, bar_g_free = bar_g + 16;
    const uint32_t bar_a = bar_g_free + 16, bar_ds = bar_a + 16, bar_fold = bar_ds + 8, bar_b = bar_fold + 16, bar_s = bar_b + 8, bar_s_free = bar_s + 8;
    const uint32_t tmem_slot = bar_s_free + 8, levels_s = bars + 256;      // sixteen floats
    static_assert(16 * C::STAGES + 16 * 4 + 8 * 4 + 4 <= 256, "barrier area");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = (int)blockIdx.x, col_tiles = p.runs.col_tiles;
    const long long t_a = p.runs.begin(cta);
    const int total = (int)(p.runs.begin(cta + 1) - t_a);
    const int rb_a = (int)(t_a / col_tiles), ct_a = (int)(t_a % col_tiles);
    // tile t of the run: its column tile and row block; true where a row block begins
    auto col_of = [&](int t) { return (ct_a + t) % col_tiles; };
    auto row_of = [&](int t) { return rb_a + (ct_a + t) / col_tiles; };
    auto new_rows = [&](int t) { return t == 0 || col_of(t) == 0; };
    // "the folds of tile t have completed": two barriers, by turns, because the folds may run two tiles ahead of the factor tiles' lane
    // where a row block begins (a phase's parity is also that of the one two before)
    auto fold_bar = [&](int t) { return bar_fold + 8u * (uint32_t)(t & 1); };
    auto fold_phase = [&](int t) { return (uint32_t)((t >> 1) & 1); };
    const int chunks = (p.b.M + kTcTok - 1) / kTcTok;
    const bool b_by_tma = (p.b.r & 7) == 0;
    const int *status = p.status;
    bool failed = false;

    if (warp == kTcTmaWarp) {
        if (lane == 0) {
            for (int s = 0; s < C::STAGES; ++s) { mbar_init(bar_full + 8 * s, 1); mbar_init(bar_empty + 8 * s, 1); }
            for (int s = 0; s < 2; ++s) { mbar_init(bar_g + 8 * s, 1); mbar_init(bar_g_free + 8 * s, kTcEpiWarps); mbar_init(bar_a + 8 * s, 1); }
            mbar_init(bar_ds, kTcEpiWarps);
            mbar_init(bar_fold, 1);
            mbar_init(bar_fold + 8, 1);
            mbar_init(bar_b, 1);
            mbar_init(bar_s, 1);
            mbar_init(bar_s_free, kTcEpiWarps);
            fence_mbar_init();
            tma_prefetch_desc(&p.tm_g);
            tma_prefetch_desc(&p.tm_x);
            tma_prefetch_desc(&p.tm_a);
        }
    } else if (warp == kTcFoldWarp) {
        tmem_alloc(tmem_slot, C::TMEM);
        tmem_relinquish();
    } else if (warp < kTcEpiWarps) {
        if (tid < 16) sts_u32(levels_s + 4 * tid, __float_as_uint(p.b.levels[tid]));
        if (!b_by_tma) {
            // rows of B that are not 16-byte multiples: element by element, zeros past rank r and past row m
            const int rr = tid >> 2, i = rb_a * kTcRows + rr;
            for (int c = 0; c < RA / 32; ++c) {
                const int chunk = (tid & 3) * (RA / 32) + c;
                uint32_t w4[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int k = chunk * 8 + 2 * e;
                    const uint32_t lo = (i < p.b.m && k < p.b.r) ? p.b.B[(size_t)i * p.b.r + k] : 0u;
                    const uint32_t hi = (i < p.b.m && k + 1 < p.b.r) ? p.b.B[(size_t)i * p.b.r + k + 1] : 0u;
                    w4[e] = lo | (hi << 16);
                }
                sts_v4(b_s + (uint32_t)((chunk >> 3) * kTcRows * 128 + (rr >> 3) * 1024 + (rr & 7) * 128 + (((chunk & 7) ^ (rr & 7)) << 4)),
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

    if (warp == kTcTmaWarp) {
        // ------------------------------------------------------------------ g and x, 64 tokens per stage
        if (lane == 0) {
            int it = 0;
            for (int t = 0; t < total && !failed; ++t) {
                const int j0 = col_of(t) * kTcCols, i0 = row_of(t) * kTcRows;
                for (int c = 0; c < chunks; ++c, ++it) {
                    const int s = it % C::STAGES;
                    if (it >= C::STAGES && !mbar_wait(bar_empty + 8 * s, (uint32_t)((it / C::STAGES - 1) & 1), status, 41)) { failed = true; break; }
                    const uint32_t bar = bar_full + 8 * s, st0 = base + (uint32_t)(s * kTcStage);
                    mbar_expect_tx(bar, (uint32_t)kTcStage);
                    tma_load_2d(st0, &p.tm_g, i0, c * kTcTok, bar);
                    tma_load_2d(st0 + kTcGAtom, &p.tm_g, i0 + 64, c * kTcTok, bar);
                    tma_load_2d(st0 + 2 * kTcGAtom, &p.tm_x, j0, c * kTcTok, bar);
                    tma_load_2d(st0 + 3 * kTcGAtom, &p.tm_x, j0 + 64, c * kTcTok, bar);
                }
            }
        }
        __syncwarp();
    } else if (warp == kTcFactorWarp) {
        // ------------------------------------------------------------------ the B tile per row block, an A tile per column tile
        if (lane == 0) {
            for (int t = 0; t < total; ++t) {
                // an A buffer is free when the folds of the tile NA before have completed, the B tile when those of the tile right before have
                if (t >= C::NA && !mbar_wait(fold_bar(t - C::NA), fold_phase(t - C::NA), status, 46)) { failed = true; break; }
                if (b_by_tma && new_rows(t)) {
                    if (t > 0 && !mbar_wait(fold_bar(t - 1), fold_phase(t - 1), status, 46)) { failed = true; break; }
                    mbar_expect_tx(bar_b, (uint32_t)C::BTILE);
                    for (int h = 0; h < RA / 64; ++h) tma_load_2d(b_s + (uint32_t)(h * kTcRows * 128), &p.tm_b, h * 64, row_of(t) * kTcRows, bar_b);
                }
                const uint32_t bar = bar_a + 8 * (t % C::NA), dst = a_s + (uint32_t)((t % C::NA) * C::ATILE);
                const int j0 = col_of(t) * kTcCols;
                mbar_expect_tx(bar, (uint32_t)(2 * p.r_pad * 128));
                tma_load_2d(dst, &p.tm_a, j0, 0, bar);
                tma_load_2d(dst + C::AATOM, &p.tm_a, j0 + 64, 0, bar);
            }
        }
        __syncwarp();
    } else if (warp == kTcMainWarp) {
        // ------------------------------------------------------------------ main MMAs
        constexpr uint32_t idesc = umma_idesc_f16(1, 1, 1, kTcRows, kTcCols);     // bf16, both operands MN-major
        const uint32_t hi = (uint32_t)(umma_desc_sw128(0, 1024, (uint32_t)kTcGAtom) >> 32);
        const uint32_t a_lo0 = (uint32_t)umma_desc_sw128(0, 1024, (uint32_t)kTcGAtom) | ((base & 0x3FFFFu) >> 4);
        const uint32_t tmem_u = warp_uniform(tmem_base), leader = elect_one();
        int it = 0, gi = 0;
        for (int t = 0; t < total && !failed; ++t) {
            int in_group = 0;                                                      // MMAs of the group so far
            for (int c = 0; c < chunks && !failed; ++c, ++it) {
                const int s = it % C::STAGES;
                if (!mbar_wait_warp(bar_full + 8 * s, (uint32_t)((it / C::STAGES) & 1), status, 42)) { failed = true; break; }
                tc_fence_after_sync();
                const uint32_t a_lo = a_lo0 + (uint32_t)((s * kTcStage) >> 4), b_lo = a_lo + (2 * kTcGAtom >> 4);
#pragma unroll
                for (int k = 0; k < kTcTok / 16; k += 2) {      // 16 tokens = 16 rows of 128 bytes
                    const int gb = gi % C::NG;
                    if (in_group == 0) {
                        if (gi >= C::NG && !mbar_wait_warp(bar_g_free + 8 * gb, (uint32_t)((gi / C::NG - 1) & 1), status, 47)) { failed = true; break; }
                        tc_fence_after_sync();
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        umma_f16_ss(tmem_u + (uint32_t)(gb * kTcCols), umma_desc_pack(a_lo + (k + h) * 128, hi), umma_desc_pack(b_lo + (k + h) * 128, hi), idesc,
                                    (in_group > 0 || h > 0) ? 1u : 0u, leader);
                    in_group += 2;
                    if (in_group == p.group || (c == chunks - 1 && k + 2 == kTcTok / 16)) {
                        umma_commit(bar_g + 8 * gb, leader);
                        ++gi;
                        in_group = 0;
                    }
                }
                umma_commit(bar_empty + 8 * s, leader);
            }
        }
    } else if (warp == kTcFoldWarp) {
        // ------------------------------------------------------------------ fold MMAs, and for QAT the scale MMA of the next tile
        const uint32_t idesc_b = umma_idesc_f16(1, 0, 0, kTcRows, 16) & ~(0x3Fu << 17) | ((uint32_t)(p.r_pad >> 3) << 17);    // dS K-major, A tile K-major
        const uint32_t idesc_a = umma_idesc_f16(1, 1, 1, kTcCols, 16) & ~(0x3Fu << 17) | ((uint32_t)(p.r_pad >> 3) << 17);    // dS MN-major, B tile MN-major
        constexpr uint32_t idesc_s = umma_idesc_f16(1, 0, 1, kTcRows, kTcCols);                                               // B tile K-major, A tile MN-major
        const uint32_t hi = (uint32_t)(umma_desc_sw128(0, 1024, 16) >> 32);
        auto desc_lo = [&](uint32_t addr, uint32_t lbo) { return (uint32_t)umma_desc_sw128(0, 1024, lbo) | ((addr & 0x3FFFFu) >> 4); };
        const uint32_t tmem_u = warp_uniform(tmem_base), leader = elect_one();
        uint32_t b_phase = 0;
        // B of a row block, before its first use
        auto wait_b = [&](int t) {
            if (!b_by_tma || !new_rows(t)) return;
            if (!mbar_wait_warp(bar_b, b_phase, status, 44)) failed = true;
            b_phase ^= 1u;
        };
        auto scale = [&](int t) {
            wait_b(t);
            if (failed) return;
            if (!mbar_wait_warp(bar_a + 8 * (t % C::NA), (uint32_t)((t / C::NA) & 1), status, 48) ||
                (t > 0 && !mbar_wait_warp(bar_s_free, (uint32_t)((t - 1) & 1), status, 49))) { failed = true; return; }
            tc_fence_after_sync();
            const uint32_t sb = desc_lo(b_s, 16), sa = desc_lo(a_s + (uint32_t)((t % C::NA) * C::ATILE), (uint32_t)C::AATOM);
            for (int k = 0; k < p.r_pad / 16; ++k)
                umma_f16_ss(tmem_u + C::S_COL, umma_desc_pack(sb + (k >> 2) * (kTcRows * 128 >> 4) + (k & 3) * 2, hi), umma_desc_pack(sa + k * 128, hi),
                            idesc_s, k > 0 ? 1u : 0u, leader);
            umma_commit(bar_s, leader);
        };
        if (QAT && total > 0 && !failed) scale(0);
        for (int t = 0; t < total && !failed; ++t) {
            const int an = t % C::NA;
            const bool ahead = C::NA == 2 && t + 1 < total && !new_rows(t + 1);       // (a new row block's B replaces the one that this tile's folds read)
            if (QAT && ahead) scale(t + 1);
            if (!QAT) wait_b(t);
            if (failed) break;
            if (!mbar_wait_warp2(bar_a + 8 * an, (uint32_t)((t / C::NA) & 1), bar_ds, (uint32_t)(t & 1), status, 50)) { failed = true; break; }
            tc_fence_after_sync();
            const uint32_t a_tile = a_s + (uint32_t)(an * C::ATILE);
            // The smallest term first, each tile onto zero: tensor cores cut sums off instead of rounding them, and this way only the largest
            // term's eight MMAs do so at the sum's size.
            const uint32_t db_col = tmem_u + C::DB_COL + (uint32_t)(p.fold_bufs == 2 && (t & 1) ? p.r_pad : 0);
            const uint32_t da_col = db_col + (uint32_t)(p.fold_bufs * p.r_pad);
            if (p.part_dB) {
                const uint32_t db = desc_lo(a_tile, 16);
#pragma unroll 1
                for (int e = 2; e >= 0; --e) {
                    const uint32_t da = desc_lo(ds0 + (uint32_t)(e * kTcDsTerm), 16);
#pragma unroll
                    for (int k = 0; k < kTcCols / 16; ++k)
                        umma_f16_ss(db_col, umma_desc_pack(da + (k >> 2) * (kTcDsAtom >> 4) + (k & 3) * 2, hi),
                                    umma_desc_pack(db + (k >> 2) * (C::AATOM >> 4) + (k & 3) * 2, hi), idesc_b, (e < 2 || k > 0) ? 1u : 0u, leader);
                }
            }
            if (p.part_dA) {
                const uint32_t db = desc_lo(b_s, (uint32_t)(kTcRows * 128));
#pragma unroll 1
                for (int e = 2; e >= 0; --e) {
                    const uint32_t da = desc_lo(ds0 + (uint32_t)(e * kTcDsTerm), (uint32_t)kTcDsAtom);
#pragma unroll
                    for (int k = 0; k < kTcRows / 16; ++k)
                        umma_f16_ss(da_col, umma_desc_pack(da + k * 128, hi), umma_desc_pack(db + k * 128, hi), idesc_a,
                                    (e < 2 || k > 0) ? 1u : 0u, leader);
                }
            }
            umma_commit(fold_bar(t), leader);
            if (QAT && !ahead && t + 1 < total) scale(t + 1);
        }
    } else {
        // ------------------------------------------------------------------ epilogue: one row of the tile and 32 columns per thread
        const int q = warp & 3, ch = warp >> 2, ri = q * 32 + lane;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const size_t row_bytes = (size_t)p.b.n * p.b.bits / 8;
        const int bits = p.b.bits;
        const uint8_t *q_end = p.b.q + (size_t)p.b.m * row_bytes;
        // where 8 columns (16 bytes) of one term of dS go: row `row` of the tile, position pos (0 .. 3) of the warp's 32 columns
        auto ds_at = [&](int row, int term, int pos) {
            return ds0 + (uint32_t)(term * kTcDsTerm + (ch >> 1) * kTcDsAtom + (row >> 3) * 1024 + (row & 7) * 128 + ((((ch & 1) * 4 + pos) ^ (row & 7)) << 4));
        };
        // a tile's contribution to dA leaves TMEM once its folds have completed (lane = column, TMEM column = rank)
        auto store_dA = [&](int t) {
            if (!p.part_dA) return;
            const int j = col_of(t) * kTcCols + ri;
            float *out = p.part_dA + (size_t)row_of(t) * p.r4 * p.b.n + j;
            const uint32_t col = C::DB_COL + (uint32_t)(p.fold_bufs * p.r_pad + (p.fold_bufs == 2 && (t & 1) ? p.r_pad : 0));
            for (int k0 = ch * 8; k0 < p.r4; k0 += 32) {          // eight ranks each: all sixteen warps have a part up to rank 32
                uint32_t v[8];
                tmem_ld_32x8(lane_addr + col + (uint32_t)k0, v);
                if (j < p.b.n)
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k0 + k < p.r4) __stcg(out + (size_t)(k0 + k) * p.b.n, __uint_as_float(v[k]));
            }
            tc_fence_before_sync();
        };
        // a tile's contribution to dB is added to this CTA's contribution to the row block, in scratch (lane = row, TMEM column = rank): only
        // this thread adds to these values, tile after tile, so the order is fixed.  (Read, added and written back, the way to L2 is waited
        // for: a fine-tuning step of 4096 x 4096 at 512 tokens 115 us
        // against 109.)
        auto store_dB = [&](int t) {
            if (!p.part_dB) return;
            const int rb = row_of(t), i = rb * kTcRows + ri;
            const bool onto = !new_rows(t);
            float *out = p.part_dB + ((size_t)(cta - p.runs.first(rb)) * p.b.m + i) * p.r4;
            const uint32_t col = C::DB_COL + (uint32_t)(p.fold_bufs == 2 && (t & 1) ? p.r_pad : 0);
            for (int k0 = ch * 16; k0 < p.r4; k0 += 64) {
                uint32_t v[16];
                tmem_ld_32x16(lane_addr + col + (uint32_t)k0, v);
                tmem_wait_ld(v);
                if (i < p.b.m)
#pragma unroll
                    for (int k = 0; k < 16; k += 4)
                        if (k0 + k < p.r4) {
                            if (onto) red_add_v4(out + k0 + k, v[k], v[k + 1], v[k + 2], v[k + 3]);
                            else __stcg(reinterpret_cast<uint4 *>(out + k0 + k), make_uint4(v[k], v[k + 1], v[k + 2], v[k + 3]));
                        }
            }
            tc_fence_before_sync();
        };
        int gi = 0;                  // groups of MMAs so far
        for (int t = 0; t < total; ++t) {
            const int i = row_of(t) * kTcRows + ri, jc = col_of(t) * kTcCols + ch * 32;
            // what does not depend on the products is requested first: the thread's codes and latent weights
            // (the last condition holds for every launch without RAGGED; left out, the loads below are scheduled worse: QAT 74 -> 80 us)
            const bool whole = i < p.b.m && jc + 32 <= p.b.n && (RAGGED || (row_bytes & 3) == 0);
            uint32_t cw[4];
            {
                const uint8_t *src = p.b.q + (whole ? (size_t)i * row_bytes + (size_t)jc * bits / 8 : 0);
                if constexpr (!RAGGED) {
#pragma unroll
                    for (int w = 0; w < 4; ++w) cw[w] = whole && w < bits ? __ldg(reinterpret_cast<const uint32_t *>(src) + w) : 0u;
                } else {
#pragma unroll
                    for (int w = 0; w < 4; ++w) cw[w] = 0u;
                    if (whole && bits == 4) load_words_anywhere<4>(src, q_end, cw);
                    else if (whole && bits == 3) load_words_anywhere<3>(src, q_end, cw);
                    else if (whole) load_words_anywhere<2>(src, q_end, cw);
                }
            }
            uint4 wq[QAT ? 4 : 1];
            if constexpr (QAT) {
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    wq[v] = make_uint4(0u, 0u, 0u, 0u);
                    if constexpr (!RAGGED) {
                        if (i < p.b.m && jc + 8 * v < p.b.n) wq[v] = __ldg(reinterpret_cast<const uint4 *>(p.b.W + (size_t)i * p.b.n + jc + 8 * v));
                    } else if (i < p.b.m && jc + 8 * v < p.b.n) {                  // n is even: 4-byte aligned
                        const uint32_t *two = reinterpret_cast<const uint32_t *>(p.b.W + (size_t)i * p.b.n + jc + 8 * v);
                        const int left = p.b.n - jc - 8 * v;
                        wq[v] = make_uint4(__ldg(two), left > 2 ? __ldg(two + 1) : 0u, left > 4 ? __ldg(two + 2) : 0u, left > 6 ? __ldg(two + 3) : 0u);
                    }
                }
            }
            float gs[32];                                                          // the tile's product, row ri, 32 columns
#pragma unroll
            for (int e = 0; e < 32; ++e) gs[e] = 0.0f;
            for (int c = 0; c < chunks * (kTcTok / 16) && !failed; c += p.group, ++gi) {
                const int b = gi % C::NG;
                if (!mbar_wait_warp(bar_g + 8 * b, (uint32_t)((gi / C::NG) & 1), status, 43)) { failed = true; break; }
                tc_fence_after_sync();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t v[16];
                    tmem_ld_32x16(lane_addr + (uint32_t)(b * kTcCols + ch * 32 + h * 16), v);
                    tmem_wait_ld(v);
#pragma unroll
                    for (int e = 0; e < 16; e += 2)
                        f32x2_split(f32x2_add(f32x2(gs[h * 16 + e], gs[h * 16 + e + 1]), f32x2(__uint_as_float(v[e]), __uint_as_float(v[e + 1]))), gs[h * 16 + e],
                                    gs[h * 16 + e + 1]);
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_g_free + 8 * b);
            }
            if (failed) break;
            if constexpr (QAT) {
                // Eq. 4: dL/dW = dL/dW^.  Eight rows at a time through the warp's own kilobyte of shared memory, so that a store covers
                // four rows' 128 bytes: a store takes the load/store unit as many cycles as it touches lines (4096 x 4096, 512 tokens: 4.5
                // thousand of a tile's 15 thousand cycles with eight rows x 32 bytes per store)
                if (p.b.dW) {
                    const uint32_t own = w_stage + (uint32_t)(warp * 1024);
                    const int ir = i - ri + q * 32, rr = lane >> 3, rc = lane & 7;
                    auto put = [&](int row, int col, uint4 o) {
                        if (row >= p.b.m || col >= p.b.n) return;
                        float *dst = p.b.dW + (size_t)row * p.b.n + col;
                        if constexpr (!RAGGED) {
                            __stcs(reinterpret_cast<uint4 *>(dst), o);
                        } else {                                                   // n is even: 8-byte aligned
                            *reinterpret_cast<uint2 *>(dst) = make_uint2(o.x, o.y);
                            if (col + 2 < p.b.n) *reinterpret_cast<uint2 *>(dst + 2) = make_uint2(o.z, o.w);
                        }
                    };
                    auto four = [&](int c) {
                        return make_uint4(__float_as_uint(gs[4 * c]), __float_as_uint(gs[4 * c + 1]), __float_as_uint(gs[4 * c + 2]), __float_as_uint(gs[4 * c + 3]));
                    };
                    if constexpr (C::WSTAGE == 0) {
#pragma unroll
                        for (int c = 0; c < 8; ++c) put(i, jc + 4 * c, four(c));
                    } else {
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            // 16-byte chunk c of row l at chunk c ^ l: neither the writes nor the reads meet in a bank
                            __syncwarp();
                            if (rr == v)
#pragma unroll
                                for (int c = 0; c < 8; ++c) sts_v4(own + (uint32_t)(rc * 128 + ((c ^ rc) << 4)), four(c));
                            __syncwarp();
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                const int l = k * 4 + rr;
                                put(ir + v * 8 + l, jc + 4 * rc, lds_v4(own + (uint32_t)(l * 128 + ((rc ^ l) << 4))));
                            }
                        }
                    }
                }
            }
            if (QAT && !mbar_wait_warp(bar_s, (uint32_t)(t & 1), status, 51)) { failed = true; break; }
            tc_fence_after_sync();
            // dS in registers: all that does not need the buffer that the folds of the tile before still read
            float d[32];
            auto level_at = [&](uint32_t code) { return __uint_as_float(lds_table(levels_s + 4u * code)); };
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t sv[QAT ? 16 : 1];
                if constexpr (QAT) tmem_ld_32x16(lane_addr + C::S_COL + (uint32_t)(ch * 32 + h * 16), sv);
                if constexpr (QAT) {
                    tmem_wait_ld(sv);
                    if (h == 1) {
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_s_free);
                    }
                }
                // the factor of dL/dS: the level, or (QAT, Eq. 5) the level minus W (/) S; 0 where S is 0
                auto factor = [&](int e, float level) -> float {
                    if constexpr (QAT) {
                        const uint4 &wv = wq[e / 8];
                        const uint32_t ww = (e % 8) / 2 == 0 ? wv.x : (e % 8) / 2 == 1 ? wv.y : (e % 8) / 2 == 2 ? wv.z : wv.w;
                        const float w = __uint_as_float((e & 1) ? (ww & 0xFFFF0000u) : (ww << 16)), sc = __uint_as_float(sv[e & 15]);
                        // w / S by a reciprocal and one residual correction: exact whenever the quotient is representable
                        // (a weight that its code reproduces exactly gets the factor 0), a rounding error otherwise
                        const float rc = rcp_approx(sc);
                        float qv = w * rc;
                        qv = fmaf(fmaf(-qv, sc, w), rc, qv);
                        return fabsf(sc) >= 1.17549435e-38f ? level - qv : 0.0f;      // (the reciprocal takes subnormal numbers for zero)
                    } else {
                        return level;
                    }
                };
                auto levels_of = [&](auto width) {         // positions of the codes inside the words are constants for each width
                    constexpr int W = decltype(width)::value;
#pragma unroll
                    for (int e = 16 * h; e < 16 * h + 16; ++e) {
                        const int bit = e * W, w = bit >> 5, sh = bit & 31;
                        uint32_t code = cw[w] >> sh;
                        if (sh + W > 32) code |= cw[w + 1 < 4 ? w + 1 : 3] << (32 - sh);
                        d[e] = gs[e] * factor(e, level_at(code & ((1u << W) - 1u)));
                    }
                };
                if (__all_sync(0xffffffffu, whole)) {
                    if (bits == 4) levels_of(std::integral_constant<int, 4>{});
                    else if (bits == 3) levels_of(std::integral_constant<int, 3>{});
                    else levels_of(std::integral_constant<int, 2>{});
                } else {
#pragma unroll
                    for (int e = 16 * h; e < 16 * h + 16; ++e)
                        d[e] = (i < p.b.m && jc + e < p.b.n) ? gs[e] * factor(e, level_at(read_code(p.b.q, row_bytes, i, jc + e, bits))) : 0.0f;
                }
            }
            // the folds of the tile before have completed: the dS buffer is free, its parts of dB and dA are in TMEM
            if (t > 0 && !mbar_wait_warp(fold_bar(t - 1), fold_phase(t - 1), status, 45)) { failed = true; break; }
            tc_fence_after_sync();
            // the three terms, eight columns (one 16-byte store each) at a time
#pragma unroll
            for (int e8 = 0; e8 < 4; ++e8) {
                uint32_t w[3][4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float a = d[8 * e8 + 2 * k], b = d[8 * e8 + 2 * k + 1];
                    const float a1 = a - __uint_as_float(__float_as_uint(a) & 0xFFFF0000u), b1 = b - __uint_as_float(__float_as_uint(b) & 0xFFFF0000u);
                    const float a2 = a1 - __uint_as_float(__float_as_uint(a1) & 0xFFFF0000u), b2 = b1 - __uint_as_float(__float_as_uint(b1) & 0xFFFF0000u);
                    w[0][k] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
                    w[1][k] = __byte_perm(__float_as_uint(a1), __float_as_uint(b1), 0x7632);
                    w[2][k] = __byte_perm(__float_as_uint(a2), __float_as_uint(b2), 0x7632);
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) sts_v4(ds_at(ri, k, e8), make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]));
            }
            // dA and dB of the tile before: with one accumulator each they have to leave before this tile's folds begin
            if (t > 0 && p.fold_bufs == 1) {
                store_dA(t - 1);
                store_dB(t - 1);
            }
            fence_proxy_async_smem();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_ds);
            if (t > 0 && p.fold_bufs == 2) {
                store_dA(t - 1);
                store_dB(t - 1);
            }
        }
        if (!__any_sync(0xffffffffu, failed) && total > 0) {
            if (!mbar_wait_warp(fold_bar(total - 1), fold_phase(total - 1), status, 45)) {
                failed = true;
            } else {
                tc_fence_after_sync();
                store_dA(total - 1);
                store_dB(total - 1);
            }
        }
    }

    if (failed) ptx::record_give_up(p.status, LORDS_ERR_TIMEOUT);
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kTcFoldWarp) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, C::TMEM);
    }
}

// A thread moves eight values, two at a time where rows are 4-byte aligned.
__global__ void lords_pad_rows_kernel(const PadJobs jobs)
{
    long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    int k = 0;
    while (k < jobs.count && e >= jobs.job[k].words) e -= jobs.job[k++].words;
    if (k == jobs.count) return;
    const PadJob &j = jobs.job[k];
    const long long row = e / (j.pitch / 8);
    const int c = (int)(e % (j.pitch / 8)) * 8;
    const uint16_t *src = j.src + row * j.cols + c;
    uint32_t w[4];
    if ((j.cols & 1) == 0) {
#pragma unroll
        for (int v = 0; v < 4; ++v) w[v] = c + 2 * v < j.cols ? __ldg(reinterpret_cast<const uint32_t *>(src) + v) : 0u;
    } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const uint32_t lo = c + 2 * v < j.cols ? __ldg(src + 2 * v) : 0u, hi = c + 2 * v + 1 < j.cols ? __ldg(src + 2 * v + 1) : 0u;
            w[v] = lo | (hi << 16);
        }
    }
    reinterpret_cast<uint4 *>(j.dst)[e] = make_uint4(w[0], w[1], w[2], w[3]);
}

// out[e] = sum over contributions t (in order) of part[t * stride + pos(e)], for dB (rows = m, inner = r, inner4 = r4:
// blocks below blocks_b) and for dA (rows = r, inner = inner4 = n: the other blocks) in one launch.  A thread has sixteen contributions on
// their way at a time (four neighbours per thread leave too few threads: 13 us instead of 10 for 4096 x 4096, r = 32, cold).
struct ReduceJob {
    const float *part;
    float *out;
    int tiles, rows, inner, inner4;
    size_t stride;
    Runs runs;            // tiles < 0: the number of contributions depends on the row block
};

__global__ void __launch_bounds__(256) lords_backward_reduce_kernel(const ReduceJob jb, const ReduceJob ja, int blocks_b)
{
    const bool isb = (int)blockIdx.x < blocks_b;
    const ReduceJob &j = isb ? jb : ja;
    const size_t e = (size_t)(isb ? blockIdx.x : blockIdx.x - blocks_b) * blockDim.x + threadIdx.x;
    griddep_wait();
    if (e >= (size_t)j.rows * j.inner) return;
    const size_t row = e / j.inner, col = e % j.inner;
    const int tiles = j.tiles >= 0 ? j.tiles : j.runs.parts((int)(row / kTcRows));
    const float *src = j.part + row * j.inner4 + col;
    float s = 0.0f;
    for (int t0 = 0; t0 < tiles; t0 += 16) {
        float v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = t0 + k < tiles ? __ldcg(src + (size_t)(t0 + k) * j.stride) : 0.0f;
#pragma unroll
        for (int k = 0; k < 16; ++k) s += v[k];
    }
    j.out[e] = s;
}

// The sums of the contributions to dB ([tiles_b][m][r4]; tiles_b < 0: see runs) and dA ([tiles_a][r4][n]); either may be absent.
int launch_reduce(const float *part_b, float *dB, int tiles_b, const Runs &runs, const float *part_a, float *dA, int tiles_a, int m, int n, int r, int r4,
                  cudaStream_t stream)
{
    ReduceJob jb = {part_b, dB, tiles_b, dB ? m : 0, r, r4, (size_t)m * r4, runs};
    ReduceJob ja = {part_a, dA, tiles_a, dA ? r : 0, n, n, (size_t)r4 * n, runs};
    const size_t nb = ((size_t)jb.rows * r + 255) / 256, na = ((size_t)ja.rows * n + 255) / 256;
    if (nb + na == 0) return LORDS_OK;
    if (nb + na > 2147483647u) return LORDS_ERR_SHAPE;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(nb + na));
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    LORDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, lords_backward_reduce_kernel, jb, ja, (int)nb));
    return LORDS_OK;
}

}  // namespace

int launch_pad_rows(const PadJobs &jobs, cudaStream_t stream)
{
    long long words = 0;
    for (int c = 0; c < jobs.count; ++c) words += jobs.job[c].words;
    if ((words + 255) / 256 > 2147483647LL) return LORDS_ERR_SHAPE;
    lords_pad_rows_kernel<<<(unsigned)((words + 255) / 256), 256, 0, stream>>>(jobs);
    LORDS_CUDA_TRY(cudaGetLastError());
    return LORDS_OK;
}

int launch_transpose_codes(const uint8_t *Q, int m, int n, int bits, uint8_t *Qt, cudaStream_t stream)
{
    const dim3 grid((unsigned)((n + kTrCols - 1) / kTrCols), (unsigned)((m + kTrRows - 1) / kTrRows));
    if (grid.y > 65535u) return LORDS_ERR_SHAPE;
    if (bits == 4) lords_transpose_codes_kernel<4><<<grid, kTrThreads, 0, stream>>>(Q, Qt, m, n);
    else if (bits == 3) lords_transpose_codes_kernel<3><<<grid, kTrThreads, 0, stream>>>(Q, Qt, m, n);
    else lords_transpose_codes_kernel<2><<<grid, kTrThreads, 0, stream>>>(Q, Qt, m, n);
    LORDS_CUDA_TRY(cudaGetLastError());
    return LORDS_OK;
}

int launch_transpose_bf16_pair(const uint16_t *src0, int rows0, int cols0, uint16_t *dst0, const uint16_t *src1, int rows1, int cols1,
                               uint16_t *dst1, cudaStream_t stream)
{
    const long long t0 = (long long)((cols0 + 31) / 32) * ((rows0 + 31) / 32), t1 = (long long)((cols1 + 31) / 32) * ((rows1 + 31) / 32);
    if (t0 + t1 > 2147483647LL) return LORDS_ERR_SHAPE;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(t0 + t1));
    cfg.blockDim = dim3(32, 8);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    LORDS_CUDA_TRY(cudaLaunchKernelEx(&cfg, lords_transpose_bf16_pair_kernel, src0, dst0, rows0, cols0, src1, dst1, rows1, cols1, (int)t0));
    return LORDS_OK;
}

template <int RA, bool QAT, bool RAGGED> static int launch_tc_variant(BwTcParams &k, const State &st, cudaStream_t stream)
{
    static bool done[kMaxDevices] = {};
    const int dev = device_slot(st);
    if (!done[dev]) {
        LORDS_CUDA_TRY(cudaFuncSetAttribute(lords_backward_tc_kernel<RA, QAT, RAGGED>, cudaFuncAttributeMaxDynamicSharedMemorySize, BwCfg<RA, QAT>::SMEM));
        done[dev] = true;
    }
    k.fold_bufs = BwCfg<RA, QAT>::DB_COL + 4 * (uint32_t)k.r_pad <= 512 ? 2 : 1;
    // (as exact as what these layers ran on before: the CUDA cores with RAGGED, the tensor cores' sum over all tokens and folds on the CUDA cores
    // without)
    const int mmas = (k.b.M + kTcTok - 1) / kTcTok * (kTcTok / 16);
    k.group = RAGGED ? (k.b.M <= 128 ? 2 : 4) : mmas <= 8 ? 4 : (mmas / 2 + 3) / 4 * 4;
    lords_backward_tc_kernel<RA, QAT, RAGGED><<<(unsigned)k.runs.ctas, kTcThreads, BwCfg<RA, QAT>::SMEM, stream>>>(k);
    LORDS_CUDA_TRY(cudaGetLastError());
    return LORDS_OK;
}

// The tensor schedule.  p.W != null: the gradients of quantisation-aware training (dW may be null).
// LORDS_ERR_UNSUPPORTED when the shapes do not suit it or the workspace cannot hold the contributions.
static int launch_backward_tc(const BwParams &p, State &st, cudaStream_t stream)
{
    const int m = p.m, n = p.n, r = p.r, M = p.M;
    BwTcParams k;
    k.b = p;
    k.r4 = (r + 3) & ~3;
    k.r_pad = (r + 15) & ~15;
    Runs &runs = k.runs;
    runs.row_blocks = (m + kTcRows - 1) / kTcRows;
    runs.col_tiles = (n + kTcCols - 1) / kTcCols;
    const long long tiles = (long long)runs.row_blocks * runs.col_tiles;
    runs.row_splits = 0;
    int parts = 1;
    if ((r & 7) == 0) {
        runs.ctas = (int)(tiles < st.sm_count ? tiles : st.sm_count);
        for (int rb = 0; rb < runs.row_blocks; ++rb) parts = runs.parts(rb) > parts ? runs.parts(rb) : parts;
    } else {
        // the least rounds of one CTA per SM times (tiles of a CTA + a fixed part worth one)
        double best = 1e30;
        for (int s = 1; s <= runs.col_tiles && s <= 64; ++s) {
            const double t = (double)(((long long)runs.row_blocks * s + st.sm_count - 1) / st.sm_count) * ((runs.col_tiles + s - 1) / s + 1.0);
            if (t < best) { best = t; runs.row_splits = s; }
        }
        parts = runs.row_splits;
        if ((long long)runs.row_blocks * parts > 2147483647LL) return LORDS_ERR_UNSUPPORTED;
        runs.ctas = runs.row_blocks * parts;
    }
    // rows of g, x or A that are not 16-byte multiples: padded copies, except where the call is so small that the CUDA cores' tiles are as
    // good (1024 x 300, two tokens)
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const int m8 = (m + 7) & ~7, n8 = (n + 7) & ~7;
    const bool pad = m8 != m || n8 != n;
    if (pad && (long long)M * m * n <= (1 << 22)) return LORDS_ERR_UNSUPPORTED;
    const size_t nb = up(p.dB ? (size_t)parts * m * k.r4 * sizeof(float) : 0), na = up(p.dA ? (size_t)runs.row_blocks * k.r4 * n * sizeof(float) : 0);
    const size_t ng = up(m8 != m ? (size_t)M * m8 * 2 : 0), nx = up(n8 != n ? (size_t)M * n8 * 2 : 0), nf = up(n8 != n ? (size_t)r * n8 * 2 : 0);
    if (nb + na + ng + nx + nf > st.workspace_bytes) return LORDS_ERR_UNSUPPORTED;
    k.part_dB = p.dB ? reinterpret_cast<float *>(st.workspace) : nullptr;
    k.part_dA = p.dA ? reinterpret_cast<float *>(st.workspace + nb) : nullptr;
    k.status = st.status_word;
    const uint16_t *g = p.g, *x = p.x, *A = p.A;
    int launches = 1;
    if (pad) {
        uint16_t *at = reinterpret_cast<uint16_t *>(st.workspace + nb + na);
        PadJobs jobs;
        jobs.count = 0;
        auto copy = [&](const uint16_t *&src, int rows, int cols, int pitch, size_t bytes) {
            if (bytes == 0) return;
            jobs.job[jobs.count++] = {src, at, cols, pitch, (long long)rows * (pitch / 8)};
            src = at;
            at += bytes / 2;
        };
        copy(g, M, m, m8, ng);
        copy(x, M, n, n8, nx);
        copy(A, r, n, n8, nf);
        const int prc = launch_pad_rows(jobs, stream);
        if (prc != LORDS_OK) return prc;
        ++launches;
    }
    if (!make_map_2d(&k.tm_g, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, g, (uint64_t)m8, (uint64_t)M, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&k.tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, x, (uint64_t)n8, (uint64_t)M, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&k.tm_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, A, (uint64_t)n8, (uint64_t)r, 64, (uint32_t)k.r_pad, CU_TENSOR_MAP_SWIZZLE_128B))
        return LORDS_ERR_CUDA;
    k.tm_b = k.tm_a;                                                       // not used where the kernel builds the B tile element by element
    if ((r & 7) == 0 &&
        !make_map_2d(&k.tm_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p.B, (uint64_t)r, (uint64_t)m, 64, (uint32_t)kTcRows, CU_TENSOR_MAP_SWIZZLE_128B))
        return LORDS_ERR_CUDA;
    int rc;
    const bool ragged = pad || (size_t)n * p.bits / 8 % 4 != 0;       // (2-bit codes: rows of 8 columns are 2 bytes)
    auto variant = [&](auto ra, auto qat) {
        constexpr int RA = decltype(ra)::value;
        constexpr bool QAT = decltype(qat)::value;
        return ragged ? launch_tc_variant<RA, QAT, true>(k, st, stream) : launch_tc_variant<RA, QAT, false>(k, st, stream);
    };
    using Small = std::integral_constant<int, 64>;
    using Large = std::integral_constant<int, 128>;
    if (p.W) rc = r <= 64 ? variant(Small{}, std::true_type{}) : variant(Large{}, std::true_type{});
    else rc = r <= 64 ? variant(Small{}, std::false_type{}) : variant(Large{}, std::false_type{});
    if (rc != LORDS_OK) return rc;
    if (p.dB || p.dA) {
        rc = launch_reduce(k.part_dB, p.dB, -1, runs, k.part_dA, p.dA, runs.row_blocks, m, n, r, k.r4, stream);
        if (rc != LORDS_OK) return rc;
        ++launches;
    }
    st.last_launches = launches;
    st.last_path = p.W ? "backward_qat_tensor" : "backward_tensor";
    return LORDS_OK;
}

int launch_backward_factors(const uint16_t *g, const uint16_t *x, const uint8_t *q, const uint16_t *B, const uint16_t *A,
                            const float *levels, int bits, int M, int m, int n, int r, float *dB, float *dA,
                            State &st, cudaStream_t stream)
{
    if (r > kRMaxBw) return LORDS_ERR_SHAPE;
    BwParams p;
    p.g = g; p.x = x; p.q = q; p.B = B; p.A = A;
    for (int c = 0; c < 16; ++c) p.levels[c] = c < (1 << bits) ? levels[c] : 0.0f;
    p.bits = bits; p.M = M; p.m = m; p.n = n; p.r = r;
    p.dB = dB; p.dA = dA;
    p.W = nullptr; p.dW = nullptr;
    int launches = 0;
    // schedule "tiles" when the workspace holds the tiles' contributions
    const int r4 = (r + 3) & ~3, it_n = (m + kT - 1) / kT, jt_n = (n + kT - 1) / kT;
    const size_t need_b = dB ? (size_t)jt_n * m * r4 * sizeof(float) : 0, need_a = dA ? (size_t)it_n * r4 * n * sizeof(float) : 0;
    // schedule "tensor": the same with 128 x 64 tiles and the tile product on the tensor cores
    if (st.forced_path == 0) {
        const int rc = launch_backward_tc(p, st, stream);
        if (rc != LORDS_ERR_UNSUPPORTED) return rc;
    }
    if (it_n <= 65535 && need_b + need_a + 256 <= st.workspace_bytes && st.forced_path != 1) {
        float *part_b = dB ? reinterpret_cast<float *>(st.workspace) : nullptr;
        float *part_a = dA ? reinterpret_cast<float *>(st.workspace + ((need_b + 255) & ~(size_t)255)) : nullptr;
        lords_backward_tile_kernel<<<dim3((unsigned)jt_n, (unsigned)it_n), kBwThreads, 0, stream>>>(p, part_b, part_a);
        LORDS_CUDA_TRY(cudaGetLastError());
        ++launches;
        {
            const int rc = launch_reduce(part_b, dB, jt_n, Runs{}, part_a, dA, it_n, m, n, r, r4, stream);
            if (rc != LORDS_OK) return rc;
            ++launches;
        }
        st.last_launches = launches;
        st.last_path = "backward_tiles";
        return LORDS_OK;
    }
    if (dB) {
        lords_backward_factors_kernel<0><<<(unsigned)((m + kT - 1) / kT), kBwThreads, 0, stream>>>(p, 0);
        LORDS_CUDA_TRY(cudaGetLastError());
        ++launches;
    }
    if (dA) {
        lords_backward_factors_kernel<1><<<(unsigned)((n + kT - 1) / kT), kBwThreads, 0, stream>>>(p, 0);
        LORDS_CUDA_TRY(cudaGetLastError());
        ++launches;
    }
    st.last_launches = launches;
    st.last_path = "backward_walk";
    return LORDS_OK;
}

// Straight-through gradients of quantisation-aware training (Eq. 4-5): the tensor schedule where the shapes
// and the workspace allow it, else the walk (any shape, no scratch memory; g^T x is formed once per
// requested factor gradient).
int launch_backward_qat(const uint16_t *g, const uint16_t *x, const uint16_t *W, const uint8_t *q, const uint16_t *B,
                        const uint16_t *A, const float *levels, int bits, int M, int m, int n, int r, float *dW, float *dB,
                        float *dA, State &st, cudaStream_t stream)
{
    if (r > kRMaxBw) return LORDS_ERR_SHAPE;
    BwParams p;
    p.g = g; p.x = x; p.q = q; p.B = B; p.A = A;
    for (int c = 0; c < 16; ++c) p.levels[c] = c < (1 << bits) ? levels[c] : 0.0f;
    p.bits = bits; p.M = M; p.m = m; p.n = n; p.r = r;
    p.dB = dB; p.dA = dA;
    p.W = W; p.dW = dW;
    if (st.forced_path == 0) {
        const int rc = launch_backward_tc(p, st, stream);
        if (rc != LORDS_ERR_UNSUPPORTED) return rc;
    }
    int launches = 0;
    const bool rows_pass = dB || !dA;                    // dL/dW alone is written by the row pass
    if (rows_pass) {
        lords_backward_factors_kernel<0><<<(unsigned)((m + kT - 1) / kT), kBwThreads, 0, stream>>>(p, dW ? 1 : 0);
        LORDS_CUDA_TRY(cudaGetLastError());
        ++launches;
    }
    if (dA) {
        lords_backward_factors_kernel<1><<<(unsigned)((n + kT - 1) / kT), kBwThreads, 0, stream>>>(p, dW && !rows_pass ? 1 : 0);
        LORDS_CUDA_TRY(cudaGetLastError());
        ++launches;
    }
    st.last_launches = launches;
    st.last_path = "backward_qat_walk";
    return LORDS_OK;
}

}  // namespace lords
