// Barriers and bulk copies, and what the kernels with eight candidates per table entry share.
#pragma once
#include <cuda.h>

#include "vl_internal.cuh"

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(unsigned long long *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok;
}
// Bulk async copy global -> this block's shared memory, completion counted on `bar`.
// dst, src 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, unsigned long long *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Tiled copy of one box of a 3-D tensor (coordinates innermost first) into this block's shared memory,
// completion counted on `bar` with the full size of the box (elements outside the tensor arrive as
// zeros).  dst 128-byte aligned; the innermost coordinate times the element size a multiple of 16.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *tm, uint32_t x, uint32_t y, uint32_t z,
                                            unsigned long long *bar, unsigned long long policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(
            smem_u32(dst)),
        "l"(tm), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}
// Tiled bulk store of one box from shared memory (elements outside the tensor are not written); completion is
// tracked by the issuing thread's bulk async-groups.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *tm, uint32_t x, uint32_t y, uint32_t z, const void *src)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                 ::"l"(tm), "r"(x), "r"(y), "r"(z), "r"(smem_u32(src))
                 : "memory");
}

// L2 policy for data that is read once: first in line for eviction, so that it does not push out what
// other kernels are about to read again.
__device__ __forceinline__ unsigned long long l2_policy_evict_first()
{
    unsigned long long policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}

// Register of candidate g in a table entry of eight.
__device__ __forceinline__ uint32_t pk8_get(const uint4 &x, int g)
{
    const uint32_t w = (g >> 1) == 0 ? x.x : ((g >> 1) == 1 ? x.y : ((g >> 1) == 2 ? x.z : x.w));
    return (g & 1) ? (w >> 16) : (w & 0xFFFFu);
}

template <int NT>
__device__ __noinline__ void rules_sweep8(const uint4 *vcons, const uint16_t *rs_prefix, const uint32_t *vinfo,
                                          const uint32_t *first_def_instr, uint32_t V, uint32_t P, const uint4 *T,
                                          uint32_t *flags, uint32_t *minR)
{
    for (uint32_t v = threadIdx.x; v < V; v += NT) {
        const uint32_t vi = vinfo[v];
        if (!(vi & VINFO_DEFINED)) continue;
        const uint4 vc = vcons[v];
        const uint32_t clo = vc.x & 0xFFFFu, chi = vc.x >> 16, al = vc.y, recip = vc.z, w = vi & 0xFFu;
        const uint4 tt = T[v];
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const uint32_t tv = pk8_get(tt, g);
            bool bad = (al > 1 && tv != __umulhi(tv, recip) * al) || tv < clo || tv + w > chi;
            if (!bad && rs_prefix) bad = rs_prefix[min(tv + w, P)] != rs_prefix[min(tv, P)];
            if (bad) {
                atomicOr(&flags[g], (uint32_t)VL_OUT_OF_RANGE);
                atomicMin(&minR[g], first_def_instr[v]);
            }
        }
    }
}

}  // namespace
