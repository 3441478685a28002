// Device-side helpers of the kernels that run on CTA pairs (cta_group::2): TMEM, MMAs, commits and loads of a pair, and the
// division of tiles among pairs.
#pragma once

#include <stdint.h>

#include "lords_ptx.cuh"

namespace lords {
namespace ptx {

__device__ __forceinline__ void tmem_alloc2(uint32_t smem_result, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// D[both CTAs' TMEM] (+)= A * B, operands in both CTAs' shared memory at the same offsets; one thread of the even CTA.
__device__ __forceinline__ void umma2_f16_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate, uint32_t leader)
{
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
        : "memory");
}
// The same with A in both CTAs' TMEM (each CTA's 128 rows) at the same address.
__device__ __forceinline__ void umma2_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate, uint32_t leader)
{
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
        : "memory");
}
// Arrive once on the barrier at this offset in both CTAs when every MMA issued so far has completed.
__device__ __forceinline__ void umma2_commit(uint32_t bar, uint32_t leader)
{
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %2, 0;\n"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n"
        "}\n" ::"r"(bar), "h"((uint16_t)3), "r"(leader)
        : "memory");
}
// A load into this CTA whose bytes are counted on a barrier of the pair's even CTA.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const void *tmap, int x, int y, uint32_t cluster_bar)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(tmap), "r"(cluster_bar), "r"(x), "r"(y) : "memory");
}

// One piece of work of a pair: k-steps [k0, k1) of a tile.
struct Piece {
    int tile, k0, k1;
};

// The pieces of pair `pair`, in order: its tiles of the whole waves, then its share of the k-steps of the tiles left over.  The
// share may begin inside a tile (that piece goes to scratch) and end inside one (the pair that begins a
// tile finishes it: it adds the other pieces, which their pairs do first).
struct Schedule {
    int next_whole, pairs, whole, ksteps;
    long long at, end;
    __device__ __forceinline__ Schedule(int pairs_, int whole_, int tiles, int ksteps_, int pair) : next_whole(pair), pairs(pairs_), whole(whole_), ksteps(ksteps_)
    {
        const long long left = (long long)(tiles - whole) * ksteps;
        at = pair * left / pairs;
        end = (pair + 1) * left / pairs;
    }
    __device__ __forceinline__ bool next(Piece &w)
    {
        if (next_whole < whole) {
            w.tile = next_whole; w.k0 = 0; w.k1 = ksteps;
            next_whole += pairs;
            return true;
        }
        if (at >= end) return false;
        const int tt = (int)(at / ksteps);
        w.tile = whole + tt;
        w.k0 = (int)(at - (long long)tt * ksteps);
        const long long stop = (long long)(tt + 1) * ksteps < end ? (long long)(tt + 1) * ksteps : end;
        w.k1 = w.k0 + (int)(stop - at);
        at = stop;
        return true;
    }
};

// Tiles that run unsplit: whole waves, less one where the tiles left over are few.  Cut into a share for every pair, a few tiles
// would be many pieces each, which their owners add up one after the other (two tiles over 74 pairs, 37 pieces each: 209 us a call
// at 14336 x 4096, 1024 tokens, where two thirds of that are due); with a wave more to cut, a tile is two or three pieces.
inline int whole_tiles(int tiles, int pairs)
{
    const int whole = tiles / pairs * pairs, left = tiles - whole;
    return left > 0 && whole > 0 && 3 * left < pairs ? whole - pairs : whole;
}

// A warp's last act on a piece.  A piece that went to scratch: one count on its flag, which is complete at `warps`.  A tile's owner:
// one count on each flag it read; the last warp leaves zero.  (No barrier among the warps: one that gave up
// would leave the others waiting.)
__device__ __forceinline__ void piece_done(int *flags, int pair, int rank, int others, bool to_scratch, int warps, int lane)
{
    if (to_scratch) {
        __threadfence();
        __syncwarp();
        if (lane == 0) asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(flags + 2 * pair + rank), "r"(1) : "memory");
    } else if (others > 0) {
        __syncwarp();
        if (lane == 0)
            for (int o = pair + 1; o <= pair + others; ++o)
                if (atomicAdd(flags + 2 * o + rank, 1) == 2 * warps - 1) flags[2 * o + rank] = 0;
    }
}

}  // namespace ptx
}  // namespace lords
