// What the kernels on CTA pairs (clusters of two, tcgen05 with cta_group::2) share.
#pragma once
#include "tc05.cuh"

namespace swimba {
namespace tc {

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Address of the same variable in the pair's first CTA, which issues the products and owns the barriers
// that the loads report to.
__device__ __forceinline__ uint32_t leader_addr(const void *p)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
    return r;
}
// Arrival at a barrier of the first CTA: rows in this SM's shared memory are ready for the pair's products (the
// products of both SMs read them where they are the second operand), tensor memory of this SM may be overwritten.
// The form is that of CUTLASS's umma_arrive_2x1SM_sm0, which announces operands written by ordinary stores of
// either CTA to products on the pair: the writes are made visible to the asynchronous proxy by the proxy fence in
// front (reads of tensor memory: completed by the tcgen05 fence), and the products read shared memory of both SMs
// through that proxy.  An arrival with a cluster-wide release and a wait with a cluster-wide acquire in its place:
// 3 x 1531 tokens of 36 heads, 16 experts, k = 4 89 -> 125 us, the gradients of 4 x 8192 790 -> 868 us.
__device__ __forceinline__ void remote_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void pair_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrives on the barrier at this offset in BOTH CTAs once all products issued so far have completed.
__device__ __forceinline__ void pair_commit(uint64_t *bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
}
// Whole-warp calls, by one warp of each CTA: all 512 columns.
__device__ __forceinline__ void pair_tmem_alloc(uint32_t *dst_smem)
{
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void pair_tmem_dealloc(uint32_t taddr)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(512) : "memory");
}
// Arrival, once this thread's cp.async copies so far have landed, that counts as one of the barrier's
// expected arrivals.
__device__ __forceinline__ void cp_async_arrive(uint64_t *bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

}  // namespace tc
}  // namespace swimba
