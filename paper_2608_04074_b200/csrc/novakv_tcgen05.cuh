// 5th-generation tensor core, TMEM, mbarrier and bulk-copy primitives of the prompt encoder (inline PTX, sm_100a).
#pragma once

#include <stdint.h>

// Bounded wait on an mbarrier phase.  Returns false when the wait has given up (or another warp of the CTA has, which
// *abort_flag in shared memory tells); the caller then stops issuing work and goes to the teardown.  The limit in clocks is
// the 64-bit number at abort_flag + MBAR_LIMIT.  Once a wait has given up the parities of this thread's later waits mean
// nothing: one may succeed on the phase before the one it wants, so what it guards has to be checked by other means.
constexpr int MBAR_LIMIT = 7;
// A try returns after a few dozen cycles whether or not the phase is over, so a polling warp takes issue slots from the
// warps it waits for: NS nanoseconds are slept between tries.
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
template <int NS>
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64(), limit = *reinterpret_cast<volatile const long long*>(abort_flag + MBAR_LIMIT);
    const int tries = limit < 64 ? (int)limit : 64;               // (a limit of 0 gives up at once)
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < tries; ++i) {
            if (NS > 0) __nanosleep(NS);
            if (mbar_try(bar, parity)) return true;
        }
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) { *abort_flag = 1; return false; }
    }
}
template <int NS = 0>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (mbar_try(bar, parity)) return true;
    return mbar_wait_slow<NS>(bar, parity, abort_flag);
}
// Wait for an MMA that has been or will be issued by this CTA whatever happens: the flag does not end it.  (After a second
// it raises the flag, after ten the MMA is given up for lost.)
__device__ __noinline__ void mbar_wait_mma_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    const long long t0 = clock64();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (mbar_try(bar, parity)) return;
        const long long t = clock64() - t0;
        if (t > 2000000000ll) *abort_flag = 1;
        if (t > 20000000000ll) return;
    }
}
__device__ __forceinline__ void mbar_wait_mma(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (!mbar_try(bar, parity)) mbar_wait_mma_slow(bar, parity, abort_flag);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(bar) : "memory");
}
// the same by lane 0 of a warp, without a branch
__device__ __forceinline__ void mbar_arrive_lane0(uint32_t bar, int lane) {
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 st;\n\tsetp.eq.s32 p, %1, 0;\n\t@p mbarrier.arrive.shared::cta.b64 st, [%0];\n\t}"
                 ::"r"(bar), "r"(lane) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(bar), "r"(bytes) : "memory");
}
// Untiled asynchronous copy from global memory, both addresses 16-byte aligned, a multiple of 16 bytes.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Tiled copy of a 2-D box (column x, row y of its first element) by a tensor map; rows beyond the tensor read as zero.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tensor_map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(tensor_map), "r"(x), "r"(y), "r"(bar) : "memory");
}
// The same box into the L2 only.
__device__ __forceinline__ void tma_prefetch_2d(const void* tensor_map, int x, int y) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tensor_map), "r"(x), "r"(y) : "memory");
}
// generic-proxy shared-memory writes become visible to the tensor core / bulk copies
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Shared-memory matrix descriptor, K-major operand.  swizzle: 0 = none (8 x 16-byte core matrices; lbo = step along K,
// sbo = step along M/N), 2 = 128-byte rows swizzled (sbo = 1024 bytes per 8 rows, lbo unused).
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo, uint32_t swizzle) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46) |
           ((uint64_t)swizzle << 61);
}
// Instruction descriptor of kind::f16, both operands K-major.  d32: binary32 accumulator (else binary16); bf16: operand type.
__host__ __device__ constexpr uint32_t umma_idesc(bool d32, bool bf16, int m, int n) {
    return (d32 ? 1u << 4 : 0u) | (bf16 ? (1u << 7) | (1u << 10) : 0u) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
// One lane of a converged warp.  (tcgen05 instructions want a uniform branch: behind `lane == 0` the MMA and the commit
// took 46 and 55 cycles to issue, behind elect.sync 6 and 34.)
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// the barrier is arrived on when all MMAs this thread issued before have completed
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

template <int COLS>
__device__ __forceinline__ void tmem_alloc(uint32_t smem_slot) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_slot), "n"(COLS) : "memory");
}
template <int COLS>
__device__ __forceinline__ void tmem_dealloc(uint32_t base) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "n"(COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
// Lane = TMEM lane (token), consecutive 32-bit columns.  The caller waits with tmem_wait_ld().
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
                   "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15]) : "r"(addr));
}
// 32 columns of binary16 accumulators, two neighbouring columns packed into a register (even column in the low half)
__device__ __forceinline__ void tmem_ld32_h2(uint32_t addr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.pack::16b.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                   "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(addr));
}
// Waits for this thread's TMEM loads.  The registers go through the wait, so that nothing reads them before it.
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                   "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]) :: "memory");
}
