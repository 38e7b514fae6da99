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

// Hardware rules on where the tuples may sit (alignment, registers of the vreg's class, reserved registers) for the eight
// candidates of a block, by its NT consumer threads, which meet on barrier BAR.  bits: room for P + 64 bits, the reserved
// registers.  All eight are checked without a branch and only a violation is looked at: with a branch per candidate and two loads
// behind it (a prefix count of the reserved registers in global memory) the sweep took 18.4 k cycles of a block with 3,301
// vregs, now 13.4 (777 rows of 11,317 instructions 93.0 us, 91.2; 4,096 of 32,000 618, 576).
template <int NT, int BAR>
__device__ __noinline__ void rules_sweep8(const uint4 *vcons, const uint16_t *rs_prefix, const uint32_t *vinfo,
                                          const uint32_t *first_def_instr, uint32_t V, uint32_t P, const uint4 *T,
                                          uint32_t *bits, uint32_t *flags, uint32_t *minR)
{
    const uint32_t tid = threadIdx.x, n_words = P / 32 + 2;  // (a range that begins at P looks at the word after it)
    for (uint32_t r = tid; r < n_words * 32; r += NT) {
        const uint32_t word = __ballot_sync(0xffffffffu, rs_prefix && r < P && rs_prefix[r + 1] != rs_prefix[r]);
        if ((tid & 31) == 0) bits[r >> 5] = word;
    }
    asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(NT) : "memory");
    uint4 vc_next = tid < V ? vcons[tid] : make_uint4(0, 0, 0, 0);
    uint32_t vi_next = tid < V ? vinfo[tid] : 0u;
    for (uint32_t v = tid; v < V; v += NT) {
        const uint4 vc = vc_next;
        const uint32_t vi = vi_next;
        if (v + NT < V) { vc_next = vcons[v + NT]; vi_next = vinfo[v + NT]; }
        if (!(vi & VINFO_DEFINED)) continue;
        const uint32_t clo = vc.x & 0xFFFFu, chi = vc.x >> 16, al = vc.y, recip = vc.z, w = vi & 0xFFu;
        const uint4 tt = T[v];
        uint32_t bad = 0;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const uint32_t tv = pk8_get(tt, g), at = min(tv, P), end = min(tv + w, P);
            // reserved registers in [at, end): up to 32 of the range lie in two words, what is wider is walked below
            const uint32_t hold = __funnelshift_r(bits[at >> 5], bits[(at >> 5) + 1], at);
            const uint32_t mask = end - at < 32 ? (1u << (end - at)) - 1u : 0xFFFFFFFFu;
            const bool b = (al > 1 && tv != __umulhi(tv, recip) * al) || tv < clo || tv + w > chi || (hold & mask);
            bad |= (b ? 1u : 0u) << g;
        }
        if (w > 32) {
#pragma unroll
            for (int g = 0; g < 8; ++g)
                for (uint32_t r = min(pk8_get(tt, g), P) + 32; r < min(pk8_get(tt, g) + w, P); ++r) bad |= ((bits[r >> 5] >> (r & 31)) & 1u) << g;
        }
        for (; bad; bad &= bad - 1) {
            const uint32_t g = __ffs(bad) - 1;
            atomicOr(&flags[g], (uint32_t)VL_OUT_OF_RANGE);
            atomicMin(&minR[g], first_def_instr[v]);
        }
    }
    asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(NT) : "memory");  // (bits may be overwritten)
}

}  // namespace
