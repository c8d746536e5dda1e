// Thin wrappers around the sm_100a PTX the tensor-core kernels are written in: mbarriers with
// bounded waits, bulk tensor copies (TMA), tcgen05 MMA / commit / tensor-memory loads, and the
// shared-memory matrix descriptor.  Shared by the single-CTA convolution kernel and the grouped
// weight-streaming kernel; everything is inline device code.
#pragma once
#include <cuda.h>
#include <stdint.h>

namespace rmsmp {

constexpr long long kWaitCycles = 2000000000LL;  // ~1 s: far beyond any legitimate wait

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// The same test with a suspend-time hint: the hardware may park the thread for up to `hint_ns`
// nanoseconds (or until the phase completes) before it answers, so a waiting thread issues an
// instruction now and then instead of spinning through the scheduler.
__device__ __forceinline__ bool mbar_try_wait_parked(uint32_t bar, uint32_t parity, uint32_t hint_ns)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity), "r"(hint_ns) : "memory");
    return ok != 0;
}
// Bounded wait built on it (same contract as mbar_wait).
__device__ __forceinline__ bool mbar_wait_parked(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                 long long limit_cycles = kWaitCycles)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 16; ++i)
            if (mbar_try_wait_parked(bar, parity, 20000u)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limit_cycles) { *abort_flag = 1; return false; }
    }
}
__device__ __forceinline__ bool mbar_wait_parked_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    bool ok = true;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait_parked(bar, parity, abort_flag);
    return __all_sync(0xffffffffu, ok);
}
// Bounded wait.  Returns false if it gave up (or another role already did).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          long long limit_cycles = kWaitCycles)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limit_cycles) { *abort_flag = 1; return false; }
    }
}
// Whole-warp form: lane 0 polls, the verdict is made uniform, and the warp-level vote orders the
// other lanes' later accesses after lane 0's observation of the barrier.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    bool ok = true;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, abort_flag);
    return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ bool mbar_wait_parked_step(uint32_t bar, uint32_t parity, volatile int* abort_flag)      // (see mbar_wait_step)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 16; ++i)
            if (__all_sync(0xffffffffu, mbar_try_wait_parked(bar, parity, 20000u))) return true;
        if (__any_sync(0xffffffffu, *abort_flag != 0 || clock64() - t0 > kWaitCycles)) { *abort_flag = 1; return false; }
    }
}
// The form of a warp that walks its loop in step: every lane polls, and the verdict is a vote, so that what follows is the
// same for the whole warp to the compiler too.
__device__ __forceinline__ bool mbar_wait_step(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if (__any_sync(0xffffffffu, *abort_flag != 0 || clock64() - t0 > kWaitCycles)) { *abort_flag = 1; return false; }
    }
}
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                            int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
        : "memory");
}
// The same with an L2 cache policy (createpolicy).
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "l"(policy)
        : "memory");
}
__device__ __forceinline__ uint64_t l2_evict_first()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_evict_normal()
{
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(map), "r"(src), "r"(c0), "r"(c1) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Fetches a descriptor, so that the first copy through it does not wait for that.
__device__ __forceinline__ void tensormap_prefetch(const CUtensorMap* m)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
}

// Shared-memory matrix descriptor: K-major rows of `row_bytes` (128 or 64) with the swizzle of that
// width; groups of 8 rows are 8*row_bytes apart.
__device__ __forceinline__ uint64_t smem_desc_kmajor(uint32_t addr, int row_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;                              // leading byte offset (unused with swizzled K-major)
    d |= (uint64_t)((8 * row_bytes) >> 4) << 32;         // stride byte offset
    d |= (uint64_t)1 << 46;                              // descriptor version of this architecture
    d |= (uint64_t)(row_bytes == 128 ? 2 : 4) << 61;     // 128-byte / 64-byte swizzle
    return d;
}
// The MMAs of a warp in step, the descriptors given as 32-bit halves of which the low one moves: all lanes take part, the elected one issues.  What a warp can issue is what bounds tiles of fewer
// than 256 columns: measured with one wait and one commit to every four MMAs, lane 0 in a branch of its own takes 124 cycles an
// MMA whatever its size; each MMA behind an election of its own 101; four behind one election 63 to 69 up to 128 columns
// and, from 160, the N / 2 that the tensor pipe takes.  (The branch, and a flag in a register as the predicate, leave the compiler in
// doubt about how many lanes issue, and operands in uniform registers out of reach.)
// One 32-code step; two (a 64-byte k-block); four (a 128-byte k-block): 32 bytes further on in both operands' rows each.
#define RMSMP_MMA_HEAD "{\n\t.reg .pred p, e;\n\t.reg .b64 da, db;\n\telect.sync _|e, 0xffffffff;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
#define RMSMP_MMA_NEXT "add.s64 da, da, 2;\n\tadd.s64 db, db, 2;\n\t"
#define RMSMP_MMA_I8(group) "@e tcgen05.mma.cta_group::" group ".kind::i8 [%0], da, db, %4, p;\n\t"
#define RMSMP_MMA_ADD "setp.eq.u32 p, 0, 0;\n\t"
template <int kSteps>
__device__ __forceinline__ void mma_i8_step(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate)
{
    static_assert(kSteps == 1 || kSteps == 2 || kSteps == 4, "");
    if (kSteps == 1)
        asm volatile(RMSMP_MMA_HEAD RMSMP_MMA_I8("1") "}" ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate) : "memory");
    else if (kSteps == 2)
        asm volatile(RMSMP_MMA_HEAD RMSMP_MMA_I8("1") RMSMP_MMA_ADD RMSMP_MMA_NEXT RMSMP_MMA_I8("1") "}"
                     ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile(RMSMP_MMA_HEAD RMSMP_MMA_I8("1") RMSMP_MMA_ADD RMSMP_MMA_NEXT RMSMP_MMA_I8("1") RMSMP_MMA_NEXT RMSMP_MMA_I8("1") RMSMP_MMA_NEXT RMSMP_MMA_I8("1") "}"
                     ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate) : "memory");
}
// One to four steps.
__device__ __forceinline__ void mma_i8_steps(int steps, uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate)
{
    if (steps == 4) {
        mma_i8_step<4>(d_tmem, a_lo, b_lo, hi, idesc, accumulate);
    } else {
        if (steps & 2) mma_i8_step<2>(d_tmem, a_lo, b_lo, hi, idesc, accumulate);
        if (steps & 1) mma_i8_step<1>(d_tmem, a_lo + 2 * (steps & 2), b_lo + 2 * (steps & 2), hi, idesc, accumulate | (uint32_t)(steps & 2));
    }
}
// Four steps of a CTA pair (256 rows, 128 in each CTA).
__device__ __forceinline__ void mma_i8_pair_step(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(RMSMP_MMA_HEAD RMSMP_MMA_I8("2") RMSMP_MMA_ADD RMSMP_MMA_NEXT RMSMP_MMA_I8("2") RMSMP_MMA_NEXT RMSMP_MMA_I8("2") RMSMP_MMA_NEXT RMSMP_MMA_I8("2") "}"
                 ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate) : "memory");
}
// Four steps with the A operand in tensor memory (8 columns a step); kFp: E3M2 x E4M3 operands and fp32 accumulators.
template <bool kFp>
__device__ __forceinline__ void mma_tmem_a_step(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t accumulate)
{
#define RMSMP_MMA_TMEM(kind, at) "@e tcgen05.mma.cta_group::1.kind::" kind " [%0], [" at "], db, %4, p;\n\tadd.s64 db, db, 2;\n\t"
#define RMSMP_MMA_TMEM4(kind) \
    asm volatile("{\n\t.reg .pred p, e;\n\t.reg .b64 db;\n\t.reg .b32 a1, a2, a3;\n\telect.sync _|e, 0xffffffff;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 db, {%2, %3};\n\t" \
                 "add.u32 a1, %1, 8;\n\tadd.u32 a2, %1, 16;\n\tadd.u32 a3, %1, 24;\n\t" \
                 RMSMP_MMA_TMEM(kind, "%1") RMSMP_MMA_ADD RMSMP_MMA_TMEM(kind, "a1") RMSMP_MMA_TMEM(kind, "a2") RMSMP_MMA_TMEM(kind, "a3") "}" \
                 ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate) : "memory")
    if (kFp) RMSMP_MMA_TMEM4("f8f6f4"); else RMSMP_MMA_TMEM4("i8");
#undef RMSMP_MMA_TMEM4
#undef RMSMP_MMA_TMEM
}
#undef RMSMP_MMA_HEAD
#undef RMSMP_MMA_NEXT
#undef RMSMP_MMA_I8
#undef RMSMP_MMA_ADD
__device__ __forceinline__ void mma_commit_step(uint32_t bar)
{
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
                 "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar) : "memory");
}
// Issue a 32-column accumulator load; the registers are valid only after tmem_ld_wait(v).
__device__ __forceinline__ void tmem_ld_issue(uint32_t taddr, uint32_t (&v)[32])
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
// Wait for the outstanding loads.  The registers pass through the statement so that no use of
// them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&v)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                   "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                   "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                   "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 :: "memory");
}

}  // namespace rmsmp
