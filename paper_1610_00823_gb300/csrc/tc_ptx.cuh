// Inline-PTX helpers for sm_103a: mbarriers, cp.async, tcgen05 (TMEM, UMMA).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vfmm {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .b64 st;\n\t"
        "mbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(bar)
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `limit` polls (returns false) so that a logic error
// ends the kernel with an error status instead of a hang.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const volatile int* abort_flag,
                                          long long limit = (1ll << 24)) {
    for (long long it = 0; it < limit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255) == 255 && *abort_flag) return false;
    }
    return false;
}

// Arrives on the mbarrier and adds `bytes` to the transaction count of its current phase.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// ---------------------------------------------------------------- bulk copies
// Plain bulk copy global -> shared of `bytes` (both addresses 16-byte aligned, bytes a multiple
// of 16), counted against the transaction count of `bar`.
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// ---------------------------------------------------------------- cp.async (16 B, L2 only)
// No memory clobber: the destination is read only after an mbarrier wait (which
// clobbers memory), and leaving it out lets the compiler batch the address loads of many copies.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes));
}
// The mbarrier receives one arrival from this thread once all its earlier cp.async copies have
// landed (.noinc: the arrival counts against the barrier's initial count).
__device__ __forceinline__ void cp_async_mbar_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Generic-proxy writes (cp.async, st.shared) -> visible to the tensor core (async proxy).
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---------------------------------------------------------------- tcgen05 / TMEM
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor (sm_100 family): start address, leading and stride
// byte offsets (16-byte units), version 1, layout type in bits 61..63.
constexpr uint64_t kLayoutSwizzle64B = 4;
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes,
                                              uint64_t layout) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (layout & 7ull) << 61;
    return d;
}

// Instruction descriptor, kind::f16: FP32 accumulate, BF16 A and B, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// MMAs and commits are issued by one elected lane of a warp whose lanes all run the issuing code with the
// same operands (elect.sync picks the same lane each time): the operands then stay in uniform registers.
// From one divergent lane an MMA takes 44.6 cycles to issue, which is more than N <= 80 needs.
//
// The A collector buffer holds the A operand of an MMA for those that follow with the same descriptor:
// the first of a run fills it, the others use it, the last one releases it, and each B operand then costs
// its own shared-memory read only. Measured per M128 x Nn x K16 MMA in the slice-product order, cycles,
// one lane without / elected lane with the collector: N = 80 52.0 / 41.6, N = 64 48.1 / 35.6,
// N = 48 44.6 / 29.5 (N / 2 at the tensor pipe's rate).
enum class CollectA { kDiscard, kFill, kUse, kLastUse };

template <CollectA kOp>
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
#define VFMM_UMMA(collect)                                                                      \
    asm volatile(                                                                               \
        "{\n\t.reg .pred p, q;\n\t"                                                            \
        "elect.sync _|q, 0xffffffff;\n\t"                                                       \
        "setp.ne.b32 p, %4, 0;\n\t"                                                             \
        "@q tcgen05.mma.cta_group::1.kind::f16" collect " [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem), \
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)                                     \
        : "memory")
    if constexpr (kOp == CollectA::kFill) VFMM_UMMA(".collector::a::fill");
    else if constexpr (kOp == CollectA::kUse) VFMM_UMMA(".collector::a::use");
    else if constexpr (kOp == CollectA::kLastUse) VFMM_UMMA(".collector::a::lastuse");
    else VFMM_UMMA("");
#undef VFMM_UMMA
}
// Arrives on the mbarrier once every tcgen05 operation issued so far by the elected lane completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}

// 32 lanes x 8 consecutive 32-bit columns, without waiting (pair with tmem_wait_ld).
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

}  // namespace tc
}  // namespace vfmm
