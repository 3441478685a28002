// Codes and scales to fp16 weights, as the scale-MMA kernels do it.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "lords_ptx.cuh"

namespace lords {
namespace ptx {

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
