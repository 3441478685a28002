// Warp-level pieces shared by the kernels that form W^ = L[Q] (.) (BA) in registers: asynchronous copies, ldmatrix,
// mma.sync and the level-pair look-up.  (Lane = 4 g + t in the fragment layouts: rows g and g + 8, columns 2t, 2t + 1.)
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "lords_ptx.cuh"

namespace lords {
namespace ptx {

// `bytes` of the 4, 8 or 16 are read, the rest is filled with zeros
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src, int bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src, int bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&v)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t (&v)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the same onto zero
__device__ __forceinline__ void mma_bf16_first(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
}
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// B[i][k], B[i][k + 1] (k even) as one word, zeros outside the matrix
__device__ __forceinline__ uint32_t load_b_pair(const uint16_t *B, int i, int k, int rows, int r)
{
    if (i >= rows || k >= r) return 0u;
    const uint16_t *src = B + (size_t)i * r + k;
    if ((r & 1) == 0) return __ldg(reinterpret_cast<const uint32_t *>(src));
    return (uint32_t)__ldg(src) | (k + 1 < r ? (uint32_t)__ldg(src + 1) << 16 : 0u);
}

// level pair (fp16x2) times a pair of scales rounded once to fp16
__device__ __forceinline__ uint32_t scaled_pair(uint32_t level, float s0, float s1)
{
    const __half2 sv = __floats2half2_rn(s0, s1);
    const __half2 wv = __hmul2(*reinterpret_cast<const __half2 *>(&level), sv);
    return *reinterpret_cast<const uint32_t *>(&wv);
}

// The 32 codes of one row's 32-column group, and the table address of a lane's pair in 8-column tile u: columns
// 8u + 2t, 8u + 2t + 1, i.e. pair 4u + t.  Table entries are 128 bytes apart.
template <int BITS> struct CodeWords {
    uint32_t w[BITS];
    __device__ __forceinline__ void read(uint32_t addr)
    {
        if constexpr (BITS == 4) {
            const uint4 v = lds_v4(addr);
            w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
        } else {
#pragma unroll
            for (int k = 0; k < BITS; ++k) w[k] = lds_u32(addr + 4 * k);
        }
    }
    __device__ __forceinline__ uint32_t address(int u, int t, uint32_t lut_lane) const
    {
        if constexpr (BITS == 4) {
            return __byte_perm(w[u], 0u, 0x4440u | (uint32_t)t) * 128u + lut_lane;            // byte t of word u
        } else if constexpr (BITS == 3) {
            // the tile's four pairs are bits 24u .. 24u + 23 of the 96; moved to bits 7 .. 30, then by 6t
            const uint32_t v = u == 0 ? w[0] << 7 : u == 1 ? __funnelshift_r(w[0], w[1], 17) : u == 2 ? __funnelshift_r(w[1], w[2], 9) : w[2] >> 1;
            return ((v >> (6 * t)) & 0x1F80u) + lut_lane;
        } else {
            const uint32_t v = (u & 1) ? w[u >> 1] >> 9 : w[u >> 1] << 7;                     // half-word u at bits 7 .. 22
            return ((v >> (4 * t)) & 0x780u) + lut_lane;
        }
    }
};

}  // namespace ptx
}  // namespace lords
