// tcgen05.cuh - inline-PTX helpers for the 5th-generation tensor cores
// (tcgen05.mma with TMEM accumulators), mbarriers and 1-D bulk copies,
// shared by the Gram kernel (gram_tc.cu) and the fused recurrence + Gram
// kernel (fused_tc.cu).  sm_100a/sm_103a only.
#pragma once

#include <stdint.h>

namespace ssm {
namespace tc {

constexpr long WAIT_LIMIT = 1L << 26;  // bounded mbarrier polls

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, no swizzle: start address, leading-dimension
// byte offset (between core matrices adjacent along K) and stride-dimension
// byte offset (between 8-element groups adjacent along M/N), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// kind::f16 instruction descriptor: D f32, A/B bf16, both MN-major, M = 128, N = n.
__device__ __forceinline__ uint32_t instr_desc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) |
           ((128u >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity) {
    for (long i = 0; i < WAIT_LIMIT; ++i)
        if (mbar_try(addr, parity)) return true;
    return false;
}

// Bounded wait that also gives up as soon as another thread of the CTA has
// recorded a failure in *fail (checked every 256 polls).
__device__ __forceinline__ bool mbar_wait_or_fail(uint32_t addr, uint32_t parity, const volatile int* fail) {
    for (long i = 0; i < WAIT_LIMIT; ++i) {
        if (mbar_try(addr, parity)) return true;
        if ((i & 255) == 255 && *fail) return false;
    }
    return false;
}

// As mbar_try, but the thread is suspended until the phase completes or about
// hint_ns nanoseconds pass, instead of returning at once: waiting warps do not
// take issue slots from the warps that work.
__device__ __forceinline__ bool mbar_try_sleep(uint32_t addr, uint32_t parity, uint32_t hint_ns) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(addr), "r"(parity), "r"(hint_ns)
        : "memory");
    return ok != 0;
}

constexpr long SLEEP_WAIT_LIMIT = 1L << 22;  // bounded suspended polls (~4 s at 1 us each)

// Bounded, suspending wait that gives up as soon as another thread of the CTA
// has recorded a failure in *fail.
__device__ __forceinline__ bool mbar_wait_sleep(uint32_t addr, uint32_t parity, const volatile int* fail) {
    for (long i = 0; i < SLEEP_WAIT_LIMIT; ++i) {
        if (mbar_try_sleep(addr, parity, 1000u)) return true;
        if (fail && *fail) return false;
    }
    return false;
}

// Non-suspending test of a phase (mbarrier.test_wait) and a bounded spin on it
// that gives up when another thread of the CTA has recorded a failure in *fail
// (checked every 1024 polls): for short hand-offs between the warps of a
// pipeline, where a suspended waiter would add its wake-up latency to every stage.
__device__ __forceinline__ bool mbar_test(uint32_t addr, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    return ok != 0;
}

constexpr long SPIN_WAIT_LIMIT = 1L << 30;  // bounded polls (seconds at the poll rate)

__device__ __forceinline__ bool mbar_spin(uint32_t addr, uint32_t parity, const volatile int* fail) {
    for (long i = 0; i < SPIN_WAIT_LIMIT; ++i) {
        if (mbar_test(addr, parity)) return true;
        if ((i & 1023) == 1023 && fail && *fail) return false;
    }
    return false;
}

__device__ __forceinline__ void mbar_init(uint64_t* m, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* m, uint32_t bytes) {
    [[maybe_unused]] uint64_t state;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 %0, [%1], %2;"
                 : "=l"(state)
                 : "r"(smem_u32(m)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* m) {
    [[maybe_unused]] uint64_t state;
    asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(state) : "r"(smem_u32(m)) : "memory");
}

// Global -> shared bulk copy (16-byte aligned addresses, size a multiple of 16),
// completion counted in bytes on mbarrier m.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint64_t* m) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(smem_u32(m))
        : "memory");
}

// Arrive on m once every tcgen05 operation issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t* m) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(m))
                 : "memory");
}

// Bounded wait, after a failure, for copies c0 .. c1 - 1 of those issued in order into a ring of
// nb barriers (at most the last nb): shared memory must not be given up with a copy on its
// way into it.  Ends at the first that does not land.
__device__ __forceinline__ void wait_copies(uint64_t* full, int nb, int c0, int c1) {
    for (int c = c0 > c1 - nb ? c0 : c1 - nb; c < c1; ++c)
        if (!mbar_wait_sleep(smem_u32(&full[c % nb]), (c / nb) & 1, nullptr)) return;
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols));
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Two 16-column loads in flight, one wait.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr + 16u));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace tc
}  // namespace ssm
