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

// (divide_tiles cuts tiles only where every pair gets steps of them: cutting has to save more than `meet` steps, so a tile has more steps than
// that, and at least a third as many tiles as pairs are cut.)
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

// The division of `tiles` tiles of `steps` steps among at most `pairs_max` CTA pairs: how many pairs, and how many tiles run unsplit,
// one per pair and wave; the steps of the others are dealt out evenly.  The pieces of a tile meet in scratch, so tiles are cut only
// where that takes more than `meet` steps off the busiest pair (4096 x 4096, 2048 tokens, 128 tiles over 74 pairs: 77 us cut, 67 in
// two waves).  Few tiles left over are cut together with a whole wave: by themselves they would be many pieces each, which their
// owners add up one after the other (two tiles over 74 pairs, 37 pieces each: 209 us a call at 14336 x 4096, 1024 tokens, where
// two thirds of that are due).
// 20: on four layer shapes at 64 to 2048 tokens, two waves against cut tiles, uncut was the faster or level where cutting saved 4 to
// 21.6 steps (by 1 to 20 %; 14336 x 4096 at 384 tokens lost 2 %), and the slower where it saved 22.5 and more.
constexpr double kMeetSteps = 20.0;      // steps of 128 columns
struct Division {
    int pairs, whole;
    double per_pair;      // steps that the busiest pair does
};
inline Division divide_tiles(int tiles, int steps, int pairs_max, int least_steps, double meet)
{
    Division d;
    const long long total = (long long)tiles * steps;
    const double uncut = (double)((tiles + pairs_max - 1) / pairs_max) * steps;
    // cut: all pairs that can be resident, but at least `least_steps` each and about four pieces to a tile
    long long pairs = total / least_steps < tiles ? tiles : total / least_steps;
    if (pairs > 4LL * tiles) pairs = 4LL * tiles;
    if (pairs > pairs_max) pairs = pairs_max;
    const double cut = (double)total / (double)pairs;
    if (uncut <= cut + meet) {
        d.pairs = tiles < pairs_max ? tiles : pairs_max;
        d.whole = tiles;
        d.per_pair = uncut;
        return d;
    }
    d.pairs = (int)pairs;
    d.whole = tiles / d.pairs * d.pairs;
    const int left = tiles - d.whole;
    if (left > 0 && d.whole > 0 && 3 * left < d.pairs) d.whole -= d.pairs;
    d.per_pair = cut;
    return d;
}

// A piece in scratch is complete: all `warps` warps of its CTA have counted on its flag.  Bounded; false if that does not come about.
__device__ __forceinline__ bool piece_ready(const int *flag, int warps, const int *status, uint32_t who, uint32_t tag)
{
    WaitLimit limit = wait_limit_start();
    for (unsigned tries = 0;; ++tries) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v >= warps) return true;
        __nanosleep(kWaitSleepNs);
        if ((tries & 63u) == 63u && wait_limit_expired(limit, status, who, 0, tag)) return false;
    }
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
