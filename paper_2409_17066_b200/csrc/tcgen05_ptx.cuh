// PTX wrappers shared by the tcgen05 kernels: mbarriers with bounded waits, linear bulk copies, shared-memory
// operand descriptors, MMA commit and fences, tensor-memory loads.
#pragma once
#include "common.cuh"

namespace vptq {
namespace tc {

constexpr unsigned long long WAIT_LIMIT_CYCLES = 4000000000ull;      // about two seconds

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred P1;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
                 "selp.b32 %0, 1, 0, P1;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Wait until the preceding kernel of the stream has completed and its writes are visible (returns at once
// when this kernel was not launched as a programmatic dependent).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bounded wait.  Returns false when the wait was abandoned (time limit here, or the abort flag raised
// elsewhere); the first to give up records VPTQ_E_TIMEOUT in the status word.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    unsigned spins = 0;
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if ((++spins & 255u) == 0) {
            if (*abort_flag) return false;
            if ((unsigned long long)(clock64() - t0) > WAIT_LIMIT_CYCLES) {
                *abort_flag = 1;
                grid_dependency_wait();                  // a preceding kernel may be the one that clears the status word
                atomicExch(status, VPTQ_E_TIMEOUT);
                return false;
            }
        }
    }
}

// One lane of a converged warp.  A warp that runs its issue loop together and lets an elected lane execute the tcgen05
// instructions keeps descriptors and barrier addresses in uniform registers; a loop that only one lane runs moves every
// operand there first, one serial move after another.
__device__ __forceinline__ bool elect_one()
{
    uint32_t is;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(is));
    return is != 0;
}
// Bounded wait for such a loop: the spin is one opaque block, so that the loop around it stays uniform for the compiler, and
// giving up only sets `gave_up` (checked by the caller where it is cheap; a wait entered with it set polls once).
__device__ __forceinline__ void mbar_wait_uniform(uint32_t bar, uint32_t parity, uint32_t &gave_up)
{
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .u64 t0, t1;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "@p bra DONE;\n\t"
                 "mov.u64 t0, %%clock64;\n\t"
                 "AGAIN:\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "@p bra DONE;\n\t"
                 "mov.u64 t1, %%clock64;\n\t"
                 "sub.u64 t1, t1, t0;\n\t"
                 "setp.lt.u64 q, t1, %3;\n\t"
                 "setp.eq.and.u32 q, %0, 0, q;\n\t"
                 "@q bra AGAIN;\n\t"
                 "mov.u32 %0, 1;\n\t"
                 "DONE:\n\t}"
                 : "+r"(gave_up) : "r"(bar), "r"(parity), "n"(WAIT_LIMIT_CYCLES) : "memory");
}

// linear bulk copy global -> shared memory (16-byte aligned addresses, size a multiple of 16)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// shared-memory operand descriptor of tcgen05.mma
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes, uint32_t layout)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);            // start address, 16-byte units
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;   // leading-dimension byte offset
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;   // stride-dimension byte offset
    d |= (uint64_t)1 << 46;                              // descriptor version of this architecture
    d |= (uint64_t)layout << 61;                         // swizzle mode
    return d;
}
constexpr uint32_t LAYOUT_SW128 = 2, LAYOUT_SW64 = 4, LAYOUT_SW32 = 6;

// Arrive on the barrier once all MMAs issued so far have completed.
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

}  // namespace tc
}  // namespace vptq
