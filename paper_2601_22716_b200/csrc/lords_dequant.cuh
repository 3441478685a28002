// Codes and scales to fp16 weights, as the scale-MMA kernels do it.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "lords_ptx.cuh"

namespace lords {
namespace ptx {

// The packed codes of one row's 64-column half of a 128-column code stage, and the table address of its code pair P (columns 2P,
// 2P + 1 of the half).  4-bit rows are 64 bytes and arrive 64-byte-swizzled (16-byte chunk c of row i sits at chunk
// c ^ ((i >> 1) & 3), which spreads the 16-byte reads of eight consecutive rows over all banks); 3-bit rows are 48 bytes, a stride that is
// conflict-free in 16-byte reads as it is (in words eight rows share a bank four ways: the half's 24 bytes are taken out of
// the 32 around them); 2-bit rows are 32 bytes.  `lut_lane`: the lane's column of a table with entries 256 bytes apart on a 64 KB
// boundary (4 bits: byte b of a word is a code pair and, as byte 1 of that address, its entry), or 128 bytes apart, table-size aligned.
template <int BITS> struct HalfRow {
    uint32_t w[2 * BITS];
    __device__ __forceinline__ void read(uint32_t qrow, int row, int ch)
    {
        if constexpr (BITS == 4) {
            const uint32_t sw = (uint32_t)((row >> 1) & 3);
            const uint4 c0 = lds_v4(qrow + (((2 * ch) ^ sw) << 4)), c1 = lds_v4(qrow + (((2 * ch + 1) ^ sw) << 4));
            w[0] = c0.x; w[1] = c0.y; w[2] = c0.z; w[3] = c0.w; w[4] = c1.x; w[5] = c1.y; w[6] = c1.z; w[7] = c1.w;
        } else if constexpr (BITS == 2) {
            const uint4 c0 = lds_v4(qrow + 16 * ch);
            w[0] = c0.x; w[1] = c0.y; w[2] = c0.z; w[3] = c0.w;
        } else {
            const uint4 c0 = lds_v4(qrow + 16 * ch), c1 = lds_v4(qrow + 16 * ch + 16);
            const uint32_t v[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
            for (int k = 0; k < 6; ++k) w[k] = ch ? v[k + 2] : v[k];
        }
    }
    __device__ __forceinline__ uint32_t address(int P, uint32_t lut_lane) const
    {
        if constexpr (BITS == 4) return __byte_perm(w[P >> 2], lut_lane, 0x7604u | (uint32_t)((P & 3) << 4));
        const int bit = 2 * BITS * P, wi = bit >> 5, off = bit & 31;
        constexpr uint32_t mask = BITS == 3 ? 0x1F80u : 0x780u;
        uint32_t sh;
        if (off + 2 * BITS > 32) sh = __funnelshift_r(w[wi], w[wi + 1 < 2 * BITS ? wi + 1 : wi], off - 7);
        else sh = off >= 7 ? (w[wi] >> (off - 7)) : (w[wi] << (7 - off));
        return (sh & mask) | lut_lane;
    }
};

// The 32 columns (chunk c of the 128-column code stage) of one row: codes -> level pairs, times the
// matching pairs of S, as 16 fp16x2 words.
template <int BITS>
__device__ __forceinline__ void dequant_chunk(uint32_t qrow, int row, int c, uint32_t lut_lane, const uint32_t (&s)[32],
                                              uint32_t (&out)[16])
{
    uint32_t lv[16];
    if constexpr (BITS == 4) {
        // 64-byte rows, 64-byte swizzle: 16-byte chunk c of row i sits at chunk c ^ ((i >> 1) & 3)
        const uint4 cw = lds_v4(qrow + (((uint32_t)c ^ (uint32_t)((row >> 1) & 3)) << 4));
        const uint32_t w[4] = {cw.x, cw.y, cw.z, cw.w};
#pragma unroll
        for (int wi = 0; wi < 4; ++wi)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                // byte b of the word is the code pair: one byte permute isolates it, one multiply-add makes
                // the address of its entry (entries are 128 bytes apart)
                const uint32_t pair = __byte_perm(w[wi], 0u, 0x4440u | (uint32_t)b);
                lv[wi * 4 + b] = lds_u32(lut_lane + pair * 128u);
            }
    } else if constexpr (BITS == 2) {
        // 32-byte rows: chunk c is the 64-bit group at byte 8c; pair p sits at bit 4p of it
        const uint32_t w[2] = {lds_u32(qrow + 8 * c), lds_u32(qrow + 8 * c + 4)};
#pragma unroll
        for (int pp = 0; pp < 16; ++pp) {
            const int off = 4 * (pp & 7);
            const uint32_t sh = off >= 7 ? (w[pp >> 3] >> (off - 7)) : (w[pp >> 3] << (7 - off));
            lv[pp] = lds_u32(lut_lane + (sh & 0x780u));
        }
    } else {
        // 48-byte rows: chunk c is the 96-bit group at byte 12c; pair p sits at bit 6p of it
        const uint32_t w[3] = {lds_u32(qrow + 12 * c), lds_u32(qrow + 12 * c + 4), lds_u32(qrow + 12 * c + 8)};
#pragma unroll
        for (int pp = 0; pp < 16; ++pp) {
            const int bit = 6 * pp, wi = bit >> 5, off = bit & 31;
            uint32_t sh;
            if (off > 26) sh = __funnelshift_r(w[wi], w[wi + 1 < 3 ? wi + 1 : 2], off - 7);
            else sh = off >= 7 ? (w[wi] >> (off - 7)) : (w[wi] << (7 - off));
            lv[pp] = lds_u32(lut_lane + (sh & 0x1F80u));
        }
    }
#pragma unroll
    for (int pp = 0; pp < 16; ++pp) {
        const __half2 sv = __floats2half2_rn(__uint_as_float(s[2 * pp]), __uint_as_float(s[2 * pp + 1]));
        const __half2 wv = __hmul2(*reinterpret_cast<const __half2 *>(&lv[pp]), sv);
        out[pp] = *reinterpret_cast<const uint32_t *>(&wv);
    }
}

}  // namespace ptx
}  // namespace lords
