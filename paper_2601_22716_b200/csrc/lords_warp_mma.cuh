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
__device__ __forceinline__ void ldmatrix_x2(uint32_t addr, uint32_t (&v)[2])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(addr) : "memory");
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
// the same onto zero, then added to d, rounded to nearest (the tensor core's own addition cuts off)
__device__ __forceinline__ void add_mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    float v[4];
    mma_bf16_first(v, a, b0, b1);
    f32x2_split(f32x2_add(f32x2(d[0], d[1]), f32x2(v[0], v[1])), d[0], d[1]);
    f32x2_split(f32x2_add(f32x2(d[2], d[3]), f32x2(v[2], v[3])), d[2], d[3]);
}
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The table of level pairs, 128 bytes an entry, one entry a thread (the first 4^BITS of the block; called by whole warps): sixteen copies of
// two fp32 values, one for each lane of a half warp, or (HALF) 32 of two fp16 values.  Stored as eight words of 16 bytes that rotate over
// the banks.  (One level a lane and two shuffles: indexed by the pair, the parameters were read again for every copy that is stored,
// sixteen addresses to a warp: 128 x 128, one token, 3.9 us a call against 2.4.)
template <int BITS, bool HALF> __device__ __forceinline__ void fill_pair_table(uint32_t table, const float (&levels)[16], int tid)
{
    const float mine = levels[tid & 15];
    const float l0 = __shfl_sync(0xffffffffu, mine, tid & ((1 << BITS) - 1)), l1 = __shfl_sync(0xffffffffu, mine, (tid >> BITS) & ((1 << BITS) - 1));
    uint4 v = make_uint4(__float_as_uint(l0), __float_as_uint(l1), __float_as_uint(l0), __float_as_uint(l1));
    if constexpr (HALF) {
        const __half2 h = __floats2half2_rn(l0, l1);
        v.x = v.y = v.z = v.w = *reinterpret_cast<const uint32_t *>(&h);
    }
    if (tid < 1 << 2 * BITS) {
#pragma unroll
        for (int k = 0; k < 8; ++k) sts_v4(table + (uint32_t)(tid * 128 + ((tid + k) & 7) * 16), v);
    }
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

// Weights held in 32 bits, multiplied by the tensor cores.  A weight is the sum of three bf16 values (8 bits of its significand
// each, exactly: the parts are cut off, not rounded), so its product with a bf16 activation is the sum of three exact
// products, over the whole range of a float.  The parts of eight weights (pairs w[k]) in the MMA's operand layout.  An infinity's lower
// parts are NaN (see add_low); the lower parts of a float below 2^-110 reach bf16's last bit.
__device__ __forceinline__ float cut_bf16(float v) { return __uint_as_float(__float_as_uint(v) & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t cut_pair(uint64_t w, uint64_t &rest)
{
    float a, b;
    f32x2_split(w, a, b);
    rest = f32x2_fma(f32x2(cut_bf16(a), cut_bf16(b)), f32x2(-1.0f, -1.0f), w);
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632u);
}
__device__ __forceinline__ void split_weights(const uint64_t (&w)[4], uint32_t (&hi)[4], uint32_t (&mid)[4], uint32_t (&lo)[4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint64_t rest, last;
        hi[k] = cut_pair(w[k], rest);
        mid[k] = cut_pair(rest, last);
        float a, b;
        f32x2_split(last, a, b);
        lo[k] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632u);
    }
}
// The sum of the lower parts' products added to that of the first parts'.  It is a NaN only where a weight is infinite or a NaN, and
// there the first parts' products have made the sum what it is.
__device__ __forceinline__ void add_low(float (&sum)[4], const float (&low)[4])
{
#pragma unroll
    for (int e = 0; e < 4; ++e) sum[e] += low[e] == low[e] ? low[e] : 0.0f;
}

// Two bf16 activations with infinities and NaNs replaced by zero: what the lower parts of a weight are multiplied by (a part that is
// zero times an infinity would make a NaN of a sum that is infinite).
__device__ __forceinline__ uint32_t finite_pair(uint32_t v)
{
    return ((v & 0x7F80u) == 0x7F80u ? 0u : v & 0xFFFFu) | ((v & 0x7F800000u) == 0x7F800000u ? 0u : v & 0xFFFF0000u);
}

// The 32 codes of one row's 32-column group; a lane's pair in 8-column tile u are columns 8u + 2t, 8u + 2t + 1, i.e. pair 4u + t.
// address: of that pair in a table of level pairs, entries 128 bytes apart.
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
    // the pair's weights in fp32: levels (a table of fp32 pairs) times scales
    __device__ __forceinline__ uint64_t weights(int u, int t, uint32_t lut_lane, uint64_t scales) const
    {
        return f32x2_mul(lds_table64(address(u, t, lut_lane)), scales);
    }
};

}  // namespace ptx
}  // namespace lords
