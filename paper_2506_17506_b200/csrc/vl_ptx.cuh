// Barriers and bulk copies, and what the kernels with eight candidates per table entry share.
#pragma once
#include <cuda.h>

#include <type_traits>

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

// The warp has read its part of a stage, or has stored its first occurrences of a tile.
__device__ __forceinline__ void warp_arrive(unsigned long long *bar)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// A thread's four columns of a tile, as eight rows have them, to "eight candidates side by side per column".
__device__ __forceinline__ void transpose8(const uint2 (&r)[8], uint4 (&pc)[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
        uint32_t w[4];
#pragma unroll
        for (int m = 0; m < 4; ++m)
            w[m] = (j < 2) ? __byte_perm(r[2 * m].x, r[2 * m + 1].x, sel) : __byte_perm(r[2 * m].y, r[2 * m + 1].y, sel);
        pc[j] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
// Those that are first occurrences (bits of first) to their table entries, off bytes into the table.
__device__ __forceinline__ void store_first8(unsigned char *table, const uint4 (&pc)[4], const uint4 &off, uint32_t first)
{
    const uint32_t of[4] = {off.x, off.y, off.z, off.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if ((first >> j) & 1) *reinterpret_cast<uint4 *>(table + of[j]) = pc[j];
}
// Every occurrence against the table (a first occurrence trivially matches; padding columns were zeroed and name the all-zero
// spare entry); o_base: the first one's column.
__device__ __forceinline__ void compare8(const unsigned char *table, const uint4 (&pc)[4], const uint4 &off, uint32_t o_base, uint32_t *flags,
                                         uint32_t *minop)
{
    const uint32_t of[4] = {off.x, off.y, off.z, off.w};
    uint4 x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = *reinterpret_cast<const uint4 *>(table + of[j]);
    uint32_t acc = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc |= (x[j].x ^ pc[j].x) | (x[j].y ^ pc[j].y) | (x[j].z ^ pc[j].z) | (x[j].w ^ pc[j].w);
    if (acc) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t d[4] = {x[j].x ^ pc[j].x, x[j].y ^ pc[j].y, x[j].z ^ pc[j].z, x[j].w ^ pc[j].w};
#pragma unroll
            for (int g = 0; g < 8; ++g)
                if ((g & 1) ? (d[g >> 1] >> 16) : (d[g >> 1] & 0xFFFFu)) {
                    atomicOr(&flags[g], (uint32_t)VL_INCONSISTENT);
                    atomicMin(&minop[g], o_base + j);
                }
        }
    }
}

// The one-hot bank nibbles of the eight candidates of a table entry (byte j: candidate j low, candidate j + 4 high): a byte
// permute looks up 1 << bank for four of them at a time.  bm: the number of banks less 1, in both halves.
__device__ __forceinline__ uint32_t bank_nibbles8(const uint32_t (&x)[4], uint32_t bm)
{
    uint32_t h[2];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        const uint32_t w = (x[2 * m] & bm) | ((x[2 * m + 1] & bm) << 8);
        h[m] = __byte_perm(0x08040201u, 0u, w | (w >> 12));
    }
    return h[0] | (h[1] << 4);
}
// 0 if all eight ranges of width w lie inside the file: with c = 0x7FFF - (P - width) added to an entry below 2^15, bit 15 of the
// sum is set iff entry + width > P; entries at or above 2^15 are outside any file these kernels accept.
__device__ __forceinline__ uint32_t outside8(const uint32_t (&x)[4], uint32_t w, uint32_t P)
{
    if (w > P) return 1u;
    const uint32_t c2 = (0x7FFFu - (P - w)) * 0x10001u;
    return (((x[0] + c2) | x[0]) | ((x[1] + c2) | x[1]) | ((x[2] + c2) | x[2]) | ((x[3] + c2) | x[3])) & 0x80008000u;
}
// Two registers with bit 15 := ((register & 31) + width > 32): the range reaches into the next word of an occupancy mask.
// 0x7FDF = 0x8000 - 33
__device__ __forceinline__ uint32_t straddle_mark(uint32_t x, uint32_t w)
{
    return (x & 0x7FFF7FFFu) | (((x & 0x001F001Fu) + w * 0x10001u + 0x7FDF7FDFu) & 0x80008000u);
}

// Bank tally of the eight candidates over the instructions with 2..4 distinct sources, by NT threads: the banks an instruction
// touches are the bits of the OR of its sources' nibbles, counted with carry-save adders and added to bank.
template <int NT>
__device__ __forceinline__ void bank_tally8(const uint32_t *Hb, const uint2 *list, const uint32_t (&seg)[4], uint32_t *bank)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    auto csa = [](uint32_t &h, uint32_t &l, uint32_t a, uint32_t b, uint32_t c) {
        const uint32_t u = a ^ b;
        h = (a & b) | (u & c);
        l = u ^ c;
    };
    // population count of each of the 8 nibbles, as byte fields: even nibbles and odd nibbles
    auto nib_even = [](uint32_t y) -> uint32_t { return y & 0x0F0F0F0Fu; };
    auto nib_odd = [](uint32_t y) -> uint32_t { return (y >> 4) & 0x0F0F0F0Fu; };
    auto nib_counts = [](uint32_t x) -> uint32_t {
        const uint32_t y = x - ((x >> 1) & 0x55555555u);
        return (y & 0x33333333u) + ((y >> 2) & 0x33333333u);
    };
    uint32_t ones = 0, twos = 0, fours = 0, acc_e = 0, acc_o = 0, rounds = 0;
    uint32_t sum[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) sum[g] = 0;
    auto flush = [&](uint32_t weight) {
#pragma unroll
        for (int g = 0; g < 8; ++g) sum[g] += weight * (((g >= 4 ? acc_o : acc_e) >> (8 * (g & 3))) & 0xFFu);
        acc_e = 0; acc_o = 0;
    };
    // one segment of the list per number of sources: as many lookups as an entry has sources (with four for every
    // entry the shared-memory pipe took 12.4 k cycles per block on 31,000 entries, now 9)
    auto segment = [&](auto sources, uint32_t e_lo, uint32_t e_hi) {
        constexpr int S = decltype(sources)::value;
        uint2 ids_next[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) ids_next[u] = e_lo + tid + u * NT < e_hi ? list[e_lo + tid + u * NT] : make_uint2(0, 0);
        for (uint32_t e0 = e_lo + tid; e0 < e_hi; e0 += 8 * NT) {
            uint2 ids[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                ids[u] = ids_next[u];
                const uint32_t en = e0 + 8 * NT + u * NT;
                ids_next[u] = en < e_hi ? list[en] : make_uint2(0, 0);
            }
            uint32_t x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                uint32_t o = Hb[ids[u].x & 0xFFFFu] | Hb[ids[u].x >> 16];
                if (S > 2) o |= Hb[ids[u].y & 0xFFFFu];
                if (S > 3) o |= Hb[ids[u].y >> 16];
                x[u] = e0 + u * NT < e_hi ? o : 0u;
            }
            uint32_t ta, tb, fa, fb, eights;
            csa(ta, ones, ones, x[0], x[1]);
            csa(tb, ones, ones, x[2], x[3]);
            csa(fa, twos, twos, ta, tb);
            csa(ta, ones, ones, x[4], x[5]);
            csa(tb, ones, ones, x[6], x[7]);
            csa(fb, twos, twos, ta, tb);
            csa(eights, fours, fours, fa, fb);
            const uint32_t c8 = nib_counts(eights);
            acc_e += nib_even(c8);
            acc_o += nib_odd(c8);
            if (++rounds == 32) {  // the byte fields hold at most 4 per round
                flush(8u);
                rounds = 0;
            }
        }
    };
    segment(std::integral_constant<int, 2>{}, seg[0], seg[1]);
    segment(std::integral_constant<int, 3>{}, seg[1], seg[2]);
    segment(std::integral_constant<int, 4>{}, seg[2], seg[3]);
    flush(8u);
    uint32_t c = nib_counts(fours);
    acc_e = nib_even(c); acc_o = nib_odd(c);
    flush(4u);
    c = nib_counts(twos);
    acc_e = nib_even(c); acc_o = nib_odd(c);
    flush(2u);
    c = nib_counts(ones);
    acc_e = nib_even(c); acc_o = nib_odd(c);
    flush(1u);
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        const uint32_t x = __reduce_add_sync(0xffffffffu, sum[g]);
        if (lane == 0 && x) atomicAdd(&bank[g], x);
    }
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
