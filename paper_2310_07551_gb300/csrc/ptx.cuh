// PTX wrappers of the digit-product kernel: bounded mbarrier waits, bulk
// copies and the tcgen05 instructions it issues.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ds_internal.h"

namespace ds {
namespace ptx {

constexpr long long kWaitCycles = 4000000000LL;   // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool bar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}
// Waits for the phase at most `limit` cycles; false when the wait gave up or
// another wait of the CTA did.  A limit below the usual one is a test's: then every
// probe returns at once, where try_wait may suspend the thread until the phase
// completes.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, long long limit)
{
    const bool at_once = limit < kWaitCycles;
    if (bar_test(bar, parity)) return true;
    const long long t0 = clock64();
    while (!(at_once ? bar_test(bar, parity) : bar_try(bar, parity))) {
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            return false;
        }
    }
    return true;
}
// One lane of a converged warp, the same each time.  A role's loop runs on the
// whole warp with only its asynchronous instructions under this predicate: the
// operands then stay in uniform registers, where a lone thread moves each of
// them there per instruction.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(p));
    return p != 0;
}
// bytes, dst and src multiples of 16
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor, K-major rows of 32 bytes in the 32-byte
// swizzle: 8-row groups 256 bytes apart
__device__ __forceinline__ uint64_t desc_sw32(uint32_t addr)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | (uint64_t)(16 >> 4) << 16 | (uint64_t)(256 >> 4) << 32 |
           (uint64_t)1 << 46 | (uint64_t)6 << 61;
}
// kind::f16 instruction descriptor, FP16 x FP16 -> FP32, both operands K-major
__device__ __forceinline__ uint32_t idesc_f16(int M, int N)
{
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D = A B + (acc ? D : 0).  KEEP: how the A operand uses the collector
// buffer: 0 not at all, 1 read and keep, 2 reuse, 3 reuse for the last time
template <int KEEP>
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
#define DS_MMA(COLL)                                                                                    \
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16" COLL \
                 " [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),                                               \
                 "l"(a), "l"(b), "r"(idesc), "r"(acc)                                                   \
                 : "memory")
    if constexpr (KEEP == 0) DS_MMA("");
    else if constexpr (KEEP == 1) DS_MMA(".collector::a::fill");
    else if constexpr (KEEP == 2) DS_MMA(".collector::a::use");
    else DS_MMA(".collector::a::lastuse");
#undef DS_MMA
}
__device__ __forceinline__ void mma_commit_to(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
}  // namespace ptx
}  // namespace ds
