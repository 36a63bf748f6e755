// Waits and issue branches of the tensor-core product kernels
// (k_matvec_tcs.cu, k_matvec_ds.cu).
#pragma once

#include <cstdint>

namespace {

constexpr long long kWaitCycles = 2000000000LL;  // ~1 s at 2 GHz
constexpr long long kTestWaitCycles = 20000;     // msd_test_expire_waits

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait.  The clock and the CTA's abort flag are only looked at once a
// first try has failed: the issuing threads wait for every stage, and what a
// satisfied wait costs is time the tensor pipe does not get back.
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_v) {
    const long long t0 = clock64();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_v) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort_v = 1;
            return false;
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_v) {
    return mbar_try(bar, parity) || mbar_wait_slow(bar, parity, abort_v);
}
// The same for copies that must land (or MMAs that must end) before the CTA
// may go on even after an abort.
__device__ __noinline__ bool mbar_settle(uint32_t bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try(bar, parity))
        if (clock64() - t0 > kWaitCycles) return false;
    return true;
}
// One thread of a converged warp, chosen so that the compiler knows the branch
// is taken by one thread: the operands of tcgen05.mma live in uniform
// registers, and under a test of the lane number every instruction is wrapped
// in a loop over its possible values (the issue loop of the digit-sliced
// product, 400 disks: 180 us that way, 132 us so).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ bool wait_unset_flag(const volatile int* flag) {
    const long long t0 = clock64();
    while (!*flag)
        if (clock64() - t0 > kTestWaitCycles) return false;
    return true;
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// global -> shared bulk copy completing on an mbarrier (16-byte aligned, size % 16 == 0)
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar));
}
// shared-memory matrix descriptor: K-major, no swizzle, given strides
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

}  // namespace
