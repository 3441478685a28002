// Thin inline-PTX wrappers for the sm_100a features the tensor-core paths use:
// mbarrier, TMA (cp.async.bulk.tensor, never with cluster multicast), tcgen05 MMA / TMEM.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace lords {
namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---- mbarrier -------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wall-clock nanoseconds, one time base for the whole GPU.
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The limit of every bounded wait.  No wait of these kernels that starts after the kernel's own
// dependency point lasts longer than the kernel itself (tens of microseconds), so a wait that has
// polled for kWaitLimitNs of wall-clock time is taken as lost; it also ends at once when the
// library's status word shows that some other role has already given up, so one give-up drains the
// whole grid instead of letting every wait run to its own limit.
constexpr unsigned long long kWaitLimitNs = 50ull * 1000 * 1000;
// ... and that has really polled for a while: a context that was merely descheduled does not count (rounds of 64 tries)
constexpr unsigned kWaitMinRounds = 64;
struct WaitLimit {
    unsigned long long g0;
    unsigned rounds;
};
__device__ __forceinline__ WaitLimit wait_limit_start()
{
    WaitLimit w;
    w.g0 = global_ns();
    w.rounds = 0;
    return w;
}
// called after every 64 unsuccessful tries; `status` is the library's device status word (may be null).
// Every 16th call it looks at the status word and at the clock (a try that fails takes 7.8 thousand cycles, about 4 us: after
// every four milliseconds of waiting).  The first wait of a grid that runs out by itself (not because the status word was already
// set) leaves a record behind the status word, for diagnosis: {tag | parity << 8 | warp << 16 |
// CTA << 32, barrier address | rounds of 64 tries << 32}.
__device__ __forceinline__ bool wait_limit_expired(WaitLimit &w, const int *status, uint32_t bar, uint32_t parity, uint32_t tag)
{
    if ((++w.rounds & 15u) != 0u) return false;
    if (status != nullptr && *reinterpret_cast<const volatile int *>(status) != 0) return true;
    if (w.rounds > kWaitMinRounds && global_ns() - w.g0 > kWaitLimitNs) {
        if (status != nullptr) {
            unsigned long long *detail = reinterpret_cast<unsigned long long *>(const_cast<int *>(status) + 2);
            const unsigned long long who = (unsigned long long)(tag & 0xFFu) | ((unsigned long long)(parity & 1u) << 8) |
                                           ((unsigned long long)((threadIdx.x >> 5) & 0xFFu) << 16) | ((unsigned long long)blockIdx.x << 32);
            if (atomicCAS(detail, 0ull, who | (1ull << 63)) == 0ull) detail[1] = (unsigned long long)bar | ((unsigned long long)w.rounds << 32);
        }
        return true;
    }
    return false;
}

// A thread that gave up a wait records it and stays about 100 us: copies and MMAs that other roles of its CTA have issued end in that
// time, before the CTA's final barrier lets its shared memory and TMEM go.
__device__ __forceinline__ void record_give_up(int *status, int code)
{
    atomicExch(status, code);
    const unsigned long long t0 = global_ns();
    for (int k = 0; k < 1000 && global_ns() - t0 < 100000ull; ++k) __nanosleep(1000);
}

// Up to 64 tries, SLEEP nanoseconds apart.  The try itself holds the thread until the phase completes or a time that the hardware sets has
// passed, so tries one after the other (SLEEP 0, four instructions each) take few issue slots and end with the phase; a sleep of 40 ns
// before each try, which ends later than the phase more often than not, cost 4096 x 1024, one token, 0.12 us of 4.25, a block of seven
// projections 73.1 us against 70.6, a rank of 128 17.3 against 16.9.  (The hint of a suspension time compiles to sleeps as well.)
// The scale-MMA kernel on CTA pairs, which runs at the power limit, keeps the sleep: 4096 x 14336, 2048 tokens, 230 us with it, 232
// without.  Level either way are the dense product (ten layers of 3 to 60 M weights, 130 to 2048 tokens) and the factor gradients,
// within 1 %.  The QAT gradients are faster without: 4096 x 4096, 512 tokens, 76.3 us and 79.3; 4096 x 14336, 256 tokens, 234 and 238.
template <int SLEEP> __device__ __forceinline__ bool mbar_try_wait_64(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    if constexpr (SLEEP == 0)
        asm volatile(
            "{\n"
            ".reg .pred p, q;\n"
            ".reg .u32 c;\n"
            "mov.u32 c, 64;\n"
            "TRY:\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "@p bra DONE;\n"
            "sub.u32 c, c, 1;\n"
            "setp.ne.u32 q, c, 0;\n"
            "@q bra TRY;\n"
            "DONE:\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    else
        asm volatile(
            "{\n"
            ".reg .pred p, q;\n"
            ".reg .u32 c;\n"
            "mov.u32 c, 64;\n"
            "TRY:\n"
            "nanosleep.u32 %3;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "@p bra DONE;\n"
            "sub.u32 c, c, 1;\n"
            "setp.ne.u32 q, c, 0;\n"
            "@q bra TRY;\n"
            "DONE:\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "n"(SLEEP)
            : "memory");
    return ok != 0;
}

// Bounded wait: gives up after kWaitLimitNs of polling (or as soon as the status word is set) and
// reports failure, so that no role of a kernel can spin forever on a shared GPU.  Callers record
// LORDS_ERR_TIMEOUT and drain.  SLEEP: 0 ordinarily; kWaitSleepNs where a measurement stands for it, and there kWaitSlackNs for producers
// that run several steps ahead.
constexpr int kWaitSleepNs = 40, kWaitSlackNs = 200;
template <int SLEEP = 0>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const int *status = nullptr, uint32_t tag = 0)
{
    if (mbar_try_wait(bar, parity)) return true;
    WaitLimit limit = wait_limit_start();
    for (;;) {
        if (mbar_try_wait_64<SLEEP>(bar, parity)) return true;
        if (wait_limit_expired(limit, status, bar, parity, tag)) return false;
    }
}

// One or several barriers for a whole warp: the tries of several overlap, where one wait after the other costs about 110 cycles
// each in a busy CTA even when every phase is long complete.  `need2` false: the third barrier is not waited for.
template <int SLEEP = 0>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar0, uint32_t par0, const int *status = nullptr, uint32_t tag = 0)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar0, par0))) return true;
    return __all_sync(0xffffffffu, mbar_wait<SLEEP>(bar0, par0, status, tag));
}
template <int SLEEP = 0>
__device__ __forceinline__ bool mbar_wait_warp2(uint32_t bar0, uint32_t par0, uint32_t bar1, uint32_t par1, const int *status = nullptr, uint32_t tag = 0)
{
    const bool a = mbar_try_wait(bar0, par0), b = mbar_try_wait(bar1, par1);
    if (__all_sync(0xffffffffu, a && b)) return true;
    return __all_sync(0xffffffffu, mbar_wait<SLEEP>(bar0, par0, status, tag) && mbar_wait<SLEEP>(bar1, par1, status, tag + 1));
}
__device__ __forceinline__ bool mbar_wait_warp3(uint32_t bar0, uint32_t par0, uint32_t bar1, uint32_t par1, uint32_t bar2, uint32_t par2, bool need2,
                                                const int *status = nullptr, uint32_t tag = 0)
{
    const bool a = mbar_try_wait(bar0, par0), b = mbar_try_wait(bar1, par1), c = !need2 || mbar_try_wait(bar2, par2);
    if (__all_sync(0xffffffffu, a && b && c)) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar0, par0, status, tag) && mbar_wait(bar1, par1, status, tag + 1) &&
                                       (!need2 || mbar_wait(bar2, par2, status, tag + 2)));
}

// ---- programmatic dependent launch ----------------------------------------------------------------
// Lets the next kernel of the stream begin (its CTAs start as resources free up).
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Returns when the previous kernel of the stream has finished and its writes are visible.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- proxies / fences -------------------------------------------------------------------------
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---- TMA ----------------------------------------------------------------------------------------
// 2-D tiled load into this CTA's shared memory; completion is counted in bytes on `bar`.
// x is the innermost coordinate (its byte offset must be a multiple of 16).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void *tmap, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tma_prefetch_desc(const void *tmap)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
}

// ---- TMEM ---------------------------------------------------------------------------------------
// One full warp allocates `cols` (power of two >= 32) TMEM columns; the base address lands in smem.
__device__ __forceinline__ void tmem_alloc(uint32_t smem_result, uint32_t cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(cols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

__device__ __forceinline__ float rcp_approx(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// 32 lanes x 32 consecutive 32-bit columns: thread l of the warp receives lane (base_lane + l).
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}
// 16 lanes x 32 consecutive fp32 columns in the accumulator layout of m16n8: for column group u of eight, v[4u], v[4u + 1] are row
// lane / 4, columns 2 (lane % 4) and + 1, v[4u + 2], v[4u + 3] the same of row lane / 4 + 8.
__device__ __forceinline__ void tmem_ld_16x32_frag(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Eight columns, complete on return.
__device__ __forceinline__ void tmem_ld_32x8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "r"(taddr)
        : "memory");
}
// The same, tied to the registers that the loads fill (16 or 32), so that nothing computed from them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                   "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                   "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 ::"memory");
}

// 32 lanes x 32 consecutive 32-bit columns, registers -> TMEM: thread l writes lane (base_lane + l).
__device__ __forceinline__ void tmem_st_32x32(uint32_t taddr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
          "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st_32x16(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---- shared-memory accesses by 32-bit shared-window address --------------------------------------
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
// An entry of a table that never changes after set-up, at an address made from loaded data.  Not volatile: volatile loads keep their
// order among themselves and with everything else that is volatile, which lines up every look-up with its use.
__device__ __forceinline__ uint32_t lds_table(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint64_t lds_table64(uint32_t addr)
{
    uint64_t v;
    asm("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 lds_v4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint4 v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts_u32(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// ---- clusters: distributed shared memory and remote mbarrier arrival ------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_nctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Address of `local_addr` (shared window of this CTA) inside CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t local_addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(rank));
    return r;
}
// Asynchronous 4-byte store into the shared memory of a CTA of the cluster; its completion is
// counted in bytes on an mbarrier of that same CTA, which also makes the value visible to whoever
// waits on the barrier: no release fence on the storing side.
__device__ __forceinline__ void st_async_cluster_f32(uint32_t cluster_addr, float v, uint32_t cluster_bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                 ::"r"(cluster_addr), "r"(__float_as_uint(v)), "r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void st_async_cluster_2f32(uint32_t addr, float a, float b, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                 ::"r"(addr), "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// The same without release at cluster scope (which costs about a thousand cycles): for what tcgen05 fences and waits
// order, that is TMEM.
__device__ __forceinline__ void mbar_arrive_pair(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded like mbar_wait, with acquire at cluster scope (the arrivals come from other CTAs).
template <int SLEEP = 0>
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, const int *status = nullptr, uint32_t tag = 0)
{
    if (mbar_try_wait_cluster(bar, parity)) return true;
    WaitLimit limit = wait_limit_start();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i) {
            if constexpr (SLEEP > 0) __nanosleep(SLEEP);
            if (mbar_try_wait_cluster(bar, parity)) return true;
        }
        if (wait_limit_expired(limit, status, bar, parity, tag)) return false;
    }
}

// ---- UMMA ---------------------------------------------------------------------------------------
// Shared-memory matrix descriptor, 128-byte swizzle.  `sbo` = byte distance between consecutive
// groups of 8 rows (K-major) / 8 K-rows (MN-major); `lbo` = byte distance between 64-element atoms
// along MN (MN-major only; ignored for K-major swizzled layouts).
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr, uint32_t sbo, uint32_t lbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;   // descriptor version for sm_100
    d |= (uint64_t)2 << 61;   // SWIZZLE_128B
    return d;
}

// A descriptor from its two 32-bit words (the start address lives in the low word, so a loop
// can step through a tile by adding byte_offset >> 4 to it).
__device__ __forceinline__ uint64_t umma_desc_pack(uint32_t lo, uint32_t hi)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
    return d;
}

// Instruction descriptor of kind::f16 (fp16 or bf16 operands of one common type, fp32 accumulate).
//   ab_format: 0 = f16, 1 = bf16.  a_mn / b_mn: 1 = that operand is MN-major in shared memory.
__host__ __device__ constexpr uint32_t umma_idesc_f16(int ab_format, int a_mn, int b_mn, int M, int N)
{
    return (1u << 4)                        // D format f32
           | ((uint32_t)ab_format << 7)     // A format
           | ((uint32_t)ab_format << 10)    // B format
           | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16)
           | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// One lane of the (converged) warp, always the same one: 1 for it, 0 for the others.
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t p;
    asm volatile("{\n.reg .pred q;\n.reg .b32 r;\nelect.sync r|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
    return p;
}
// A value that is the same in every lane, in a form that the compiler knows to be: operands of the instructions
// below then live in uniform registers.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// The tcgen05 instructions of an issuing warp are executed by the whole converged warp under a predicate that is true for one lane
// (`leader`, from elect_one) instead of inside a branch that one lane takes: in the branch every operand of every
// instruction goes through a move from a vector to a uniform register, and one thread issued an MMA per 57
// cycles whatever its size; under the predicate they leave at the tensor core's rate (128 x 16 x 16: 12 cycles, 128 x 32
// x 16: 17, measured on an idle SM).  All operands must be the same in every lane.
//
// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void umma_f16_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate, uint32_t leader)
{
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate, uint32_t leader)
{
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "setp.ne.b32 q, %5, 0;\n"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n" ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
        : "memory");
}
// Arrive once on `bar` when every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar, uint32_t leader)
{
    asm volatile(
        "{\n"
        ".reg .pred q;\n"
        "setp.ne.b32 q, %1, 0;\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(bar), "r"(leader)
        : "memory");
}

// Two fp32 values in one 64-bit register: one instruction issued for both.
__device__ __forceinline__ uint64_t f32x2(float lo, float hi)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void f32x2_split(uint64_t v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t f32x2_mul(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t f32x2_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t f32x2_add(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

}  // namespace ptx
}  // namespace lords
