// The whole check of eight candidates by one thread block out of shared memory.
//
// The batched kernels (vl_verify.cu) hand a candidate's table from kernel to kernel through global memory: four launches, of
// which each leaves part of the device idle, and 1.2 times the bytes of the rows.  Here the block that streams eight rows
// keeps their table (16 bytes per vreg, eight registers side by side) until the verdicts are written:
//   1. the rows stream through a ring in shared memory; table from the first occurrences, Consistency;
//   2. a sweep over the vregs: Realizability (file and rules), bank nibbles, marks of ranges that straddle a mask word;
//   3. the bank tally;
//   4. Safety: eight lanes, one per candidate, take a chunk of the walk and apply its events to occupancy masks of their own
//      (column `tid` of [word][thread]), starting from the masks of the block's through-set;
//   5. a candidate with a collision: the exact counts, by the whole block, or (HAND) left to k_exact.
// A vreg at or beyond P takes part in step 4 as if it sat at P: two of them live together then collide, so that a chunk is
// never missed, and step 5 compares the true registers.
#include <algorithm>
#include <type_traits>

#include "vl_exact.cuh"
#include "vl_ptx.cuh"

#define E_STAGES 4
#define E_BAR 1  // the barrier of the consumer warps

namespace {

// Where the parts of a block's shared memory start (bytes): the table, then the region that is the copy ring, then the bank
// nibbles, then the occupancy masks, then the arrays of the exact counts; the through-set masks at the region's end.
struct ESmem {
    uint32_t region, th, misc, coll, ex_w, ex_cv, ex_coll, ex_list, cb, NS, total;
};

struct EMisc {
    unsigned long long bar[E_STAGES], empty[E_STAGES];  // a stage is full; every consumer warp has read it
    unsigned long long stored[2];                       // every consumer warp has stored its first occurrences of a tile (by tile parity)
    unsigned long long never;                           // test hook: nothing completes it
    uint32_t flags[8], minop[8], minR[8], bank[8], nout[8], thcol[8];
    uint32_t pairs[8], mind[8];
    uint32_t any, marks, abort_flag, next;
    FMisc f;
};

struct EParams {
    FParams f;
    ESmem sm;
    uint32_t nOp8, ntiles, nC, CW, bank_total, pf;
    uint32_t test_wait;  // test hook: the consumers wait on a barrier that nothing completes, with a short limit
    const uint4 *opoff;
    const uint8_t *first4;
    const uint32_t *ev8, *cev_off, *chunk_blk, *short_chunk;
    uint32_t *status;
};
template <int N>
struct EMany {
    EParams p[N];
};
static_assert(sizeof(EMany<VL_EIGHT_MANY>) <= 32764, "kernel arguments");

__device__ __forceinline__ void bulk_g2s_hint(void *dst, const void *src, uint32_t bytes, unsigned long long *bar, unsigned long long policy)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
                 : "memory");
}
__device__ __forceinline__ uint32_t atom_xor(uint32_t addr, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.shared.xor.b32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
    return old;
}
// The same where v is not 0; else 0.
__device__ __forceinline__ uint32_t atom_xor_some(uint32_t addr, uint32_t v, uint32_t some)
{
    uint32_t old = 0;
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n @p atom.shared.xor.b32 %0, [%1], %2;\n}\n" : "+r"(old) : "r"(addr), "r"(v), "r"(some) : "memory");
    return old;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}

// Eight events at ev for one candidate (see the walk in k_eight), some of whose ranges reach into the next word: an atomic more,
// in the order of the events.  The occupied bits that tests found.  A function of its own: in the walk's loop it slowed the other
// events down.  (Rows of which no tuple is aligned, with a load, a change and a store for each word one after the other / with
// atomics, us: 2,000 instructions, 1,600 rows 42.1 / 35.6; 8,000, 1,184 rows 72.1 / 62.2; 24,000, 600 rows 143 / 124.)
template <int NT>
__device__ __noinline__ uint32_t apply_far(const uint32_t *ev, uint32_t entry, uint32_t occ_addr)
{
    uint32_t viol = 0;
    uint32_t w[8], t[8];
    {
        const uint4 a = reinterpret_cast<const uint4 *>(ev)[0], b = reinterpret_cast<const uint4 *>(ev)[1];
        w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = lds_u16(entry + (w[u] & EV8_OFFSET));
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
        uint32_t lo[4], hi[4], old_hi[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t x = w[h + u], mask = x >> EV8_MASK_SHIFT, keep = x & EV8_HOLD ? 0u : 0xFFFFFFFFu;
            const uint32_t at = occ_addr + (t[h + u] & 0x7FE0u) * (NT / 8);
            lo[u] = __funnelshift_l(0u, mask, t[h + u]);
            hi[u] = __funnelshift_l(mask, 0u, t[h + u]);
            t[h + u] = atom_xor(at, lo[u] & keep);
            old_hi[u] = atom_xor_some(at + NT * 4, hi[u] & keep, hi[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (w[h + u] & EV8_TEST) viol |= (t[h + u] & lo[u]) | (old_hi[u] & hi[u]);
    }
    return viol;
}

// NT consumer threads and a producer warp; 256 threads leave room for two blocks per multiprocessor (three, with 72 registers
// and a ring of three stages: 6,400 rows of 64 programs 355 us with liveness, 334 with two).  HAND: candidates with a collision
// are left to k_exact, which spreads their counts over all multiprocessors.
template <int NT, int N, bool HAND>
__global__ void __launch_bounds__(NT + 32, NT == 256 ? 2 : 1) k_eight(const __grid_constant__ EMany<N> a)
{
    constexpr int G = 8;
    constexpr uint32_t TILE = NT * 4;  // columns per tile and candidate: four per thread
    constexpr uint32_t ROW_BYTES = TILE * 2, STAGE_BYTES = ROW_BYTES * G, WARPS = NT / 32;
    const EParams &e = a.p[N == 1 ? 0 : blockIdx.y];
    const FParams &q = e.f;
    const uint64_t k0 = (uint64_t)blockIdx.x * G;
    if (N > 1 && k0 >= q.K) return;
    extern __shared__ __align__(128) unsigned char smem[];
    uint4 *T = reinterpret_cast<uint4 *>(smem);  // [V + 1]
    unsigned char *region = smem + e.sm.region;
    uint32_t *Hb = reinterpret_cast<uint32_t *>(region);         // [V] bank nibbles
    uint32_t *s_th = reinterpret_cast<uint32_t *>(smem + e.sm.th);    // [nB][Wp][8]
    uint32_t *s_coll = reinterpret_cast<uint32_t *>(smem + e.sm.coll);  // [8][CW] chunks that collided
    EMisc *M = reinterpret_cast<EMisc *>(smem + e.sm.misc);
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid < G) {
        M->flags[tid] = 0; M->minop[tid] = 0xFFFFFFFFu; M->minR[tid] = 0xFFFFFFFFu; M->bank[tid] = 0; M->nout[tid] = 0;
        M->thcol[tid] = 0; M->pairs[tid] = 0; M->mind[tid] = 0xFFFFFFFFu;
    }
    if (tid == 0) {
        M->any = 0; M->marks = 0; M->abort_flag = 0; M->next = 0;
        for (uint32_t s = 0; s < E_STAGES; ++s) { mbar_init(&M->bar[s], 1); mbar_init(&M->empty[s], WARPS); }
        mbar_init(&M->stored[0], WARPS);
        mbar_init(&M->stored[1], WARPS);
        mbar_init(&M->never, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        T[q.V] = make_uint4(0, 0, 0, 0);  // the spare entry: what padding columns are compared with
    }
    for (uint32_t j = tid; j < G * e.CW; j += NT + 32) s_coll[j] = 0;
    pdl_go();
    __syncthreads();
    pdl_wait();  // (the rows, and what liveness computed)

    auto wait_bar = [&](unsigned long long *bar, uint32_t parity) {
        // Bounded.  When it runs out the block raises the status bit and carries on with short waits to the end of the
        // streaming phase, where it leaves; the producer issues no further copies.
        if (mbar_try_wait(bar, parity)) return;
        uint32_t spins = 0;
        const uint32_t limit = *(volatile uint32_t *)&M->abort_flag ? 64u : (1u << 20);
        while (!mbar_try_wait(bar, parity)) {
            if (++spins > limit) {
                M->abort_flag = 1;
                atomicOr(e.status, ST_DEVICE_WAIT);
                break;
            }
        }
    };
    if (tid >= NT) {  // ------------------------------------------------------------ producer warp: a lane per row
        const uint16_t *row = q.cand + min(k0 + (lane & 7), q.K - 1) * q.pitch;
        const unsigned long long stream_once = l2_policy_evict_first();
        uint32_t issued = 0, stage = 0, parity = 0;
        for (uint32_t t = 0; t < e.ntiles; ++t) {
            if (t >= e.sm.NS) {  // the stage still holds tile t - NS: wait until the consumer warps have read it
                if (lane == 0) wait_bar(&M->empty[stage], parity ^ 1u);
                if (__shfl_sync(0xffffffffu, *(volatile uint32_t *)&M->abort_flag, 0)) break;
            }
            issued = t + 1;
            const uint32_t bytes = min(TILE, e.nOp8 - t * TILE) * 2;
            if (lane == 0) mbar_expect_tx(&M->bar[stage], bytes * G);
            __syncwarp();
            if (lane < G) bulk_g2s_hint(region + (size_t)stage * STAGE_BYTES + lane * ROW_BYTES, row + (size_t)t * TILE, bytes, &M->bar[stage], stream_once);
            if (++stage == e.sm.NS) { stage = 0; parity ^= 1; }
        }
        __syncwarp();
        // No thread block goes away while a copy into its shared memory is on its way: not even if a consumer's wait runs out
        // after the last copy has been issued.
        if (lane == 0)
            for (uint32_t s = 0; s < e.sm.NS && s < issued; ++s) {
                const uint32_t t_last = s + (issued - 1 - s) / e.sm.NS * e.sm.NS;  // the last tile issued into stage s
                uint32_t spins = 0;
                while (!mbar_try_wait(&M->bar[s], (t_last / e.sm.NS) & 1u) && ++spins < (1u << 20)) {}
            }
        return;  // (from here on the consumer warps meet on a barrier of their own)
    }
    {   // ---------------------------------------------------------------------- 1. the rows (see k_tables8)
        const uint32_t spare_off = q.V * 16u;
        const uint4 *opoff = e.opoff + tid;
        const uint8_t *first4 = e.first4 + tid;
        auto compare = [&](const uint4 (&pc)[4], const uint4 &off, uint32_t o_base) { compare8(smem, pc, off, o_base, M->flags, M->minop); };
        uint32_t stage = 0, parity = 0;
        const uint32_t last = e.ntiles - 1;
        // thread i asks for line i % (ROW_BYTES / 128) of row i / (ROW_BYTES / 128) of a tile further ahead into L2
        const unsigned char *pf_ptr = nullptr;
        if (e.pf && tid < G * (ROW_BYTES / 128))
            pf_ptr = reinterpret_cast<const unsigned char *>(q.cand + min(k0 + tid / (ROW_BYTES / 128), q.K - 1) * q.pitch) +
                     (tid % (ROW_BYTES / 128)) * 128;
        uint4 off_n = opoff[0], off_n2 = opoff[NT];
        uint32_t first_n = first4[0], first_n2 = first4[NT];
        // one tile: load and transpose, store first occurrences, compare the tile before
        auto step = [&](uint32_t t, uint4 (&pc)[4], uint4 &off, const uint4 (&ppc)[4], const uint4 &poff, auto is_last) {
            constexpr bool LAST = decltype(is_last)::value;
            off = off_n;
            const uint32_t first = first_n;
            off_n = off_n2;
            first_n = first_n2;
            if (!LAST) {
                off_n2 = opoff[(size_t)(t + 2) * NT];
                first_n2 = first4[(size_t)(t + 2) * NT];
                if (pf_ptr && t + e.pf < last) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf_ptr + (size_t)(t + e.pf) * ROW_BYTES));
            }
            wait_bar(&M->bar[stage], parity);
            uint2 r[G];
            const unsigned char *src = region + (size_t)stage * STAGE_BYTES + tid * 8;
#pragma unroll
            for (int g = 0; g < G; ++g) r[g] = *reinterpret_cast<const uint2 *>(src + g * ROW_BYTES);
            transpose8(r, pc);
            if (!LAST) {
                warp_arrive(&M->empty[stage]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)  // columns beyond the rows compare as zero against the spare entry
                    if (t * TILE + tid * 4 + j >= q.nO) pc[j] = make_uint4(0, 0, 0, 0);
            }
            store_first8(smem, pc, off, first);
            warp_arrive(&M->stored[t & 1]);
            if (t) wait_bar(&M->stored[(t - 1) & 1], ((t - 1) >> 1) & 1u);
            compare(ppc, poff, (t - 1) * TILE + tid * 4);
            if (++stage == e.sm.NS) { stage = 0; parity ^= 1; }
        };
        uint4 pcA[4], pcB[4], offA, offB;
#pragma unroll
        for (int j = 0; j < 4; ++j) pcB[j] = make_uint4(0, 0, 0, 0);
        offB = make_uint4(spare_off, spare_off, spare_off, spare_off);  // "the tile before tile 0": zeros against the spare entry
        const std::integral_constant<bool, false> more{};
        if (e.test_wait) {  // test hook: this wait runs out
            uint32_t spins = 0;
            while (!mbar_try_wait(&M->never, 0)) {
                if (++spins > (1u << 16)) { M->abort_flag = 1; atomicOr(e.status, ST_DEVICE_WAIT); break; }
            }
        }
        uint32_t t = 0;
        for (; t + 2 <= last; t += 2) {
            step(t, pcA, offA, pcB, offB, more);
            step(t + 1, pcB, offB, pcA, offA, more);
        }
        if (t < last) {  // an odd number of tiles before the last: keep "the tile before" in B
            step(t, pcA, offA, pcB, offB, more);
#pragma unroll
            for (int j = 0; j < 4; ++j) pcB[j] = pcA[j];
            offB = offA;
        }
        step(last, pcA, offA, pcB, offB, std::integral_constant<bool, true>{});
        wait_bar(&M->stored[last & 1], (last >> 1) & 1u);
        compare(pcA, offA, last * TILE + tid * 4);
    }
    bar_all<NT, E_BAR>();
    // A wait ran out: copies that are still on their way may land in what takes the ring's place from here on (lists of
    // instructions among it), and the table may hold anything.  The rows get a record that is no verdict.  (If a wait of the
    // producer runs out, so does one of every consumer, for the tile that is never issued: all threads see the same flag.)
    if (M->abort_flag) {
        if (tid < G && k0 + tid < q.K) {
            if (HAND) q.ex.items[k0 + tid] = 0;
            q.out[k0 + tid] = vl_verdict{0u, -1, 0u, 0u};
        }
        return;
    }

    // ---- 2. one sweep over the vregs (see k_tables8)
    load_blocks(q, &M->f);
    for (uint32_t j = tid; q.use_th && j < q.nB * q.Wp * G; j += NT) s_th[j] = 0;
    // (the sweep below changes table entries)
    if (q.vcons) rules_sweep8<NT, E_BAR>(q.vcons, q.rs_prefix, q.vinfo, q.first_def_instr, q.V, q.P, T, Hb, M->flags, M->minR);
    {
        uint32_t mk = 0;
        const uint32_t bm = (q.B - 1) * 0x10001u;
        uint32_t vis_next[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) vis_next[u] = tid + u * NT < q.V ? q.vinfo[tid + u * NT] : 0u;
        for (uint32_t v0 = tid; v0 < q.V; v0 += 4 * NT) {
            uint32_t vis[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                vis[u] = vis_next[u];
                const uint32_t vn = v0 + 4 * NT + u * NT;
                vis_next[u] = vn < q.V ? q.vinfo[vn] : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t v = v0 + u * NT, vi = vis[u];
                if (v >= q.V) break;
                const uint4 tt = T[v];
                uint32_t x[4] = {tt.x, tt.y, tt.z, tt.w};
                Hb[v] = bank_nibbles8(x, bm);
                if (!(vi & VINFO_OCCURS)) continue;
                const uint32_t w = vi & 0xFFu, f = outside8(x, w, q.P);
                if (f) {
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        const uint32_t tv = (g & 1) ? x[g >> 1] >> 16 : x[g >> 1] & 0xFFFFu;
                        if (tv + w > q.P) {
                            if (vi & VINFO_DEFINED) {
                                atomicOr(&M->flags[g], (uint32_t)VL_OUT_OF_RANGE);
                                atomicMin(&M->minR[g], q.first_def_instr[v]);
                            }
                            M->nout[g] = 1;
                            if (tv > q.P) x[g >> 1] = (g & 1) ? (x[g >> 1] & 0xFFFFu) | (q.P << 16) : (x[g >> 1] & 0xFFFF0000u) | q.P;
                        }
                    }
                }
                uint32_t o[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) o[m] = straddle_mark(x[m], w);
                if ((o[0] ^ tt.x) | (o[1] ^ tt.y) | (o[2] ^ tt.z) | (o[3] ^ tt.w)) T[v] = make_uint4(o[0], o[1], o[2], o[3]);
                mk |= o[0] | o[1] | o[2] | o[3];
            }
        }
        if (__any_sync(0xffffffffu, mk & 0x80008000u) && lane == 0) M->marks = 1;
    }
    bar_all<NT, E_BAR>();

    // ---- 4a. the masks of the through-sets: a warp per program block, eight lanes per member
    const uint32_t smem_base = smem_u32(smem);
    for (uint32_t b = warp; q.use_th && b < q.nB; b += WARPS) {
        constexpr int TU = 4;  // members in flight
        const uint32_t g = lane & 7, j1 = M->f.th_off[b + 1];
        uint32_t *mask = s_th + b * q.Wp * G + g;
        bool hit = false;
        for (uint32_t j0 = M->f.th_off[b] + (lane >> 3); j0 < j1; j0 += 4 * TU) {
            uint32_t x[TU];
#pragma unroll
            for (int u = 0; u < TU; ++u) x[u] = q.th[min(j0 + u * 4, j1 - 1)];
#pragma unroll
            for (int u = 0; u < TU; ++u) {
                if (j0 + u * 4 >= j1) break;
                const uint32_t pos = lds_u16(smem_base + (x[u] & 0xFFFFu) * 16 + g * 2) & 0x7FFFu;
                const unsigned long long m = (unsigned long long)((1u << (x[u] >> 16)) - 1u) << (pos & 31);  // (widths of at most 8)
                hit |= (atomicOr(mask + (pos >> 5) * G, (uint32_t)m) & (uint32_t)m) != 0;
                if (m >> 32) hit |= (atomicOr(mask + (pos >> 5) * G + G, (uint32_t)(m >> 32)) & (uint32_t)(m >> 32)) != 0;
            }
        }
        if (hit) atomicOr(&M->thcol[g], 1u << b);  // through-sets are used only if nB <= 32
    }
    // ---- 3. bank tally over the instructions with 2..4 distinct sources
    bank_tally8<NT>(Hb, q.bank_list, q.bank_seg, M->bank);
    bar_all<NT, E_BAR>();  // (the bank nibbles make room for the masks)

    // ---- 4b. the walk: a warp takes four chunks, eight lanes each.  Bound by the shared-memory pipe (an atomic per candidate and
    // event, 2.2 cycles a warp; load, change and store take 3.6) and, where there are few chunks, by a warp's chain of them.  Two
    // candidates per lane share the lookups but halve the warps: 6,400 rows of 64 programs 344 us against 331.
    {
        uint32_t *occ = reinterpret_cast<uint32_t *>(region) + tid;  // words NT apart
        const uint32_t g_own = lane & 7, g2 = g_own * 2, none = e.cev_off[e.nC];  // (no-ops lie behind the last chunk)
        const uint32_t occ_addr = smem_u32(occ);
        const bool check = M->marks != 0;
        for (;;) {
            uint32_t first = 0;
            if (lane == 0) first = atomicAdd(&M->next, 4u);
            first = __shfl_sync(0xffffffffu, first, 0);
            if (first >= e.nC) break;
            const uint32_t c = first + (lane >> 3);
            const uint32_t e0 = c < e.nC ? e.cev_off[c] : 0u, e1 = c < e.nC ? e.cev_off[c + 1] : 0u;  // (multiples of 8 events)
            const uint32_t n_max = __reduce_max_sync(0xffffffffu, e1 - e0);
            uint4 xa, xb;
            auto fetch = [&](uint32_t at) {
                const uint4 *p = reinterpret_cast<const uint4 *>(e.ev8 + (at < e1 ? at : none));
                xa = p[0];
                xb = p[1];
            };
            fetch(e0);
            if (q.use_th && c < e.nC) {
                const uint32_t *src = s_th + e.chunk_blk[c] * q.Wp * G + g_own;
                for (uint32_t wd = 0; wd < q.Wp; ++wd) occ[wd * NT] = src[wd * G];
            } else {
                for (uint32_t wd = 0; wd < q.Wp; ++wd) occ[wd * NT] = 0;
            }
            __syncwarp();
            uint32_t viol = 0;
            // Eight events at a time; the next eight are on their way, and the line after those of the next (a line holds 32 events
            // of a chunk) is asked for.  Toggling returns the old word: occupied and released are both a toggle as long as no
            // collision has been seen (after one, the chunk is counted exactly anyway).
            auto events = [&](auto marked) {
#pragma unroll 1
                for (uint32_t i = 0; i < n_max; i += 8) {
                    const uint32_t w[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
                    if (e0 + i + 64 < e1) asm volatile("prefetch.global.L1 [%0];" ::"l"(e.ev8 + e0 + i + 64));
                    fetch(e0 + i + 8);
                    uint32_t t[8], m[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) t[u] = *reinterpret_cast<const uint16_t *>(smem + ((w[u] & EV8_OFFSET) | g2));
                    if (decltype(marked)::value && __any_sync(0xffffffffu, (t[0] | t[1] | t[2] | t[3] | t[4] | t[5] | t[6] | t[7]) & 0x8000u)) {
                        viol |= apply_far<NT>(e.ev8 + (e0 + i < e1 ? e0 + i : none), smem_base + g2, occ_addr);
                        continue;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        m[u] = __funnelshift_l(0u, w[u] >> EV8_MASK_SHIFT, t[u]);
                        t[u] = atom_xor(occ_addr + (t[u] & 0x7FE0u) * (NT / 8), w[u] & EV8_HOLD ? 0u : m[u]);
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (w[u] & EV8_TEST) viol |= t[u] & m[u];
                }
            };
            if (check) events(std::integral_constant<bool, true>{});
            else events(std::integral_constant<bool, false>{});
            if (viol) {
                atomicOr(&s_coll[g_own * e.CW + (c >> 5)], 1u << (c & 31));
                atomicOr(&M->any, 1u << g_own);
            }
        }
    }
    bar_all<NT, E_BAR>();

    // ---- 5. exact counts of the candidates with a collision, one after the other
    for (uint32_t g = 0; !HAND && g < G; ++g) {
        if (k0 + g >= q.K || !(((M->any >> g) & 1u) | M->thcol[g])) continue;
        uint16_t *X = reinterpret_cast<uint16_t *>(region);
        uint8_t *W = region + e.sm.ex_w;
        uint32_t *cv = reinterpret_cast<uint32_t *>(region + e.sm.ex_cv), *coll = reinterpret_cast<uint32_t *>(region + e.sm.ex_coll);
        uint2 *list = reinterpret_cast<uint2 *>(region + e.sm.ex_list);
        const uint16_t *row = q.cand + (k0 + g) * q.pitch;
        const uint32_t out_of_file = M->nout[g];
        for (uint32_t v = tid; v <= q.V; v += NT) {
            uint32_t t = reinterpret_cast<const uint16_t *>(T + v)[g] & 0x7FFFu;
            if (out_of_file && t == q.P && v < q.V) {  // (it may lie beyond)
                const uint32_t pos = q.first_occ[v];
                t = pos != 0xFFFFFFFFu ? row[pos] : 0u;
            }
            X[v] = (uint16_t)t;
            W[v] = v < q.V ? (uint8_t)q.vinfo[v] : (uint8_t)0;
        }
        for (uint32_t s = tid; s < ((q.nS + 31u) & ~31u); s += NT) {  // a chunk that collided marks its short chunks
            const uint32_t c = e.short_chunk[min(s, q.nS - 1)];
            const uint32_t bits = __ballot_sync(0xffffffffu, s < q.nS && ((s_coll[g * e.CW + (c >> 5)] >> (c & 31)) & 1u));
            if (lane == 0) coll[s >> 5] = bits;
        }
        if (tid == 0) {
            M->f.bank = M->f.pairs = 0;
            M->f.mind = 0xFFFFFFFFu;
            M->f.thcol = M->thcol[g];
        }
        bar_all<NT, E_BAR>();
        exact_counts<NT, false, false, E_BAR>(q, X, W, cv, coll, list, &M->f, 0, 1, row);
        uint32_t n = 0;  // the bank tally, exactly: sources may share a register
        for (uint32_t j = tid; j < q.bank_seg[3]; j += NT)
            n += bank_entry(q.bank_list[j], j < q.bank_seg[1] ? 2u : (j < q.bank_seg[2] ? 3u : 4u), X, q.B - 1);
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0 && n) atomicAdd(&M->f.bank, n);
        bar_all<NT, E_BAR>();
        if (tid == 0) {
            M->pairs[g] = M->f.pairs;
            M->mind[g] = M->f.mind;
            M->bank[g] = e.bank_total - M->f.bank;  // (as the others leave it)
        }
        bar_all<NT, E_BAR>();
    }

    // ---- the verdicts, a warp per candidate
    if (warp < G && k0 + warp < q.K) {
        const uint32_t g = warp, o = M->minop[g];
        uint32_t first = min(M->minR[g], M->mind[g]);
        if (o != 0xFFFFFFFFu) {
            uint32_t i;
            if (q.entry_instr) {
                // dictionary rows: entries are in block order and, inside a block, in order of first occurrence, so the
                // lowest violating entry is also the lowest violating instruction
                i = q.entry_instr[o];
            } else {  // operand -> instruction: the last i with op_off[i] <= operand, 32 probes per round
                uint32_t lo = 0, hi = q.nI;  // op_off[lo] <= o < op_off[hi]
                while (hi - lo > 1) {
                    const uint32_t step = (hi - lo + 31) / 32, at = min(lo + (lane + 1) * step, hi);
                    const uint32_t below = __popc(__ballot_sync(0xffffffffu, q.op_off[at] <= o));  // (op_off ascends)
                    const uint32_t nlo = min(lo + below * step, hi);
                    hi = min(nlo + step, hi);
                    lo = nlo;
                }
                i = lo;
            }
            first = min(first, i);
        }
        if (HAND && (((M->any >> g) & 1u) | M->thcol[g])) {
            const uint64_t k = k0 + g;
            uint32_t chunks = 0;
            for (uint32_t w = lane; w < e.CW; w += 32) {
                const uint32_t bits = s_coll[g * e.CW + w];
                q.ex.anom[k * e.CW + w] = bits;
                chunks += __popc(bits);
            }
            chunks = __reduce_add_sync(0xffffffffu, chunks);
            const bool full = chunks == e.nC;  // (with every chunk counted in full, nothing is left of the through-sets)
            const uint32_t thcol = full ? 0u : M->thcol[g];
            if (thcol) chunks += e.nC / 8;  // (the sources in the through-set)
            if (lane < 4) q.ex.racc[k * 4 + lane] = 0;
            if (lane == 0) {
                uint32_t *cs = q.ex.cstate + k * 8;
                cs[CS_FLAGS] = M->flags[g]; cs[CS_FIRST] = first; cs[CS_BANK] = e.bank_total - M->bank[g];
                cs[CS_WALK] = ((M->any >> g) & 1u ? WALK_ANOM : 0u) | (full ? WALK_FULL : 0u); cs[CS_THCOL] = thcol;
                q.ex.items[k] = exact_parts(chunks, EXACT_PART_CHUNKS) | exact_parts(chunks, EXACT_FINE_CHUNKS) << 16;
            }
            return;
        }
        if (lane == 0) {
            if (HAND) q.ex.items[k0 + g] = 0;
            const uint32_t flags = M->flags[g] | (M->pairs[g] ? (uint32_t)VL_INTERFERENCE : 0u);
            vl_verdict vd;
            vd.flags = flags ? flags : (uint32_t)VL_PASS;
            vd.first_violation_instr = first == 0xFFFFFFFFu ? -1 : (int32_t)first;
            vd.conflict_pairs = M->pairs[g];
            vd.bank_conflicts = e.bank_total - M->bank[g];
            q.out[k0 + g] = vd;
        }
    }
}

inline uint32_t up(uint64_t x, uint32_t n) { return (uint32_t)((x + n - 1) / n * n); }

// Shared memory of a block with NT consumer threads; total = 0 if it does not fit the budget.
ESmem eight_smem(const vl_program *p, uint32_t NT, uint32_t budget)
{
    ESmem s{};
    const uint32_t Wp = (p->P + p->wmax + 31) / 32, stage = NT * 64;
    const uint64_t table = ((uint64_t)p->V + 1) * 16;
    const uint64_t th = p->use_th ? (uint64_t)p->nB * Wp * 32 : 0u, coll = (uint64_t)8 * ((p->nC + 31) / 32) * 4;
    const uint64_t counts = ((uint64_t)p->P + p->wmax + 2) * 4;  // (of one program block, see exact_counts)
    s.ex_w = up((p->V + 1) * 2ull, 16);
    s.ex_coll = up(s.ex_w + (p->V + 1ull), 16);
    s.ex_list = up(s.ex_coll + (p->nS + 31) / 32 * 4ull + 4, 16);
    s.ex_cv = up(s.ex_list + p->nS * 8ull, 16);
    const uint64_t exact = s.ex_cv + (p->use_th ? counts : 0u);
    const uint64_t masks = std::max<uint64_t>((p->V + 1) * 4ull, (uint64_t)Wp * NT * 4) + th;
    const uint64_t least = up(std::max<uint64_t>(2ull * stage, std::max(exact, masks)), 128);
    const uint64_t rest = up(table, 128) + up(sizeof(EMisc), 16) + up(coll, 16);
    if (rest + least > budget) return s;
    s.region = up(table, 128);
    s.NS = (uint32_t)std::min<uint64_t>(E_STAGES, (budget - rest) / stage);
    const uint32_t region = (uint32_t)std::max<uint64_t>(least, (uint64_t)s.NS * stage);
    s.th = s.region + region - (uint32_t)th;
    s.cb = p->use_th ? (uint32_t)std::min<uint64_t>(p->nB, (region - s.ex_cv) / counts) : p->nB;
    s.misc = s.region + region;
    s.coll = s.misc + up(sizeof(EMisc), 16);
    s.total = s.coll + up(coll, 16);
    return s;
}

struct EPlan {
    uint32_t NT;  // 0: does not fit
    ESmem sm;
};
#define E_HALF (227u * 1024 / 2 - 1024)
// Two blocks of 256 threads per multiprocessor where the rows give it that many and the tables let them, else one of 512.
EPlan eight_plan(vl_program *p, uint64_t K)
{
    EPlan pl{};
    if (K > 8ull * vl_sm_count(p)) {
        pl.sm = eight_smem(p, 256, E_HALF);
        if (pl.sm.total) { pl.NT = 256; return pl; }
    }
    pl.sm = eight_smem(p, 512, 227u * 1024);
    if (pl.sm.total) { pl.NT = 512; return pl; }
    pl.sm = eight_smem(p, 256, 227u * 1024);
    if (pl.sm.total) pl.NT = 256;
    return pl;
}

template <int NT, int N, bool HAND>
cudaError_t launch_eight(int device, const EMany<N> &many, dim3 grid, uint32_t smem, cudaStream_t st)
{
    const cudaError_t e = allow_smem<k_eight<NT, N, HAND>, 227 * 1024>(device);
    if (e != cudaSuccess) return e;
    return launch_overlap(k_eight<NT, N, HAND>, grid, NT + 32, smem, st, true, many);
}
}  // namespace

// What does not depend on the rows (nor on the layout): the table offsets of the events fit their words, widths their masks,
// and register numbers stay below the mark.
bool vl_eight_takes(const vl_program *p) { return p->V < 16384 && p->wmax <= 8 && p->P + p->wmax <= 32768u && p->nC > 0; }

// Up to one block per multiprocessor it wins over the batched kernels for every program it takes, beyond that up to about 24
// million instructions times rows and 16,000 instructions: the batched kernels look an event up for 64 rows at a time.  This
// kernel / the batched ones, us, 10 % of the rows failing: 2,000 instructions, 1,184 rows 37 / 49, 2,368 rows 42 / 100, 4,736 rows
// 70 / 103, 12,000 rows 146 / 151; 8,000 instructions, 600 rows 62 / 83, 1,184 rows 66 / 92, 2,368 rows 90 / 152, 3,000 rows
// 142 / 164; 11,900 instructions, 1,600 rows 102 / 115, 2,001 rows 103 / 114; 14,500 instructions, 1,420 rows 116 / 115, 1,550 rows 116 / 119;
// 18,000 instructions, 1,330 rows 150 / 139; 32,000 instructions, 1,184 rows 133 / 158; 64 and 1,000 instructions, 10,000
// rows 53 / 87 and 103 / 126, 375,000 and 24,000 rows 1,550 / 1,969 and 215 / 230.  With 40 % failing: 8,000 instructions, 1,600
// rows 122 / 138, 3,000 rows 177 / 198.
// Little more than one block per multiprocessor leaves most of them with one block of 256 threads: up to 1 1/6 of them the
// line lies at 11,000 instructions.  1,190 rows, none failing and 10 %: 10,000 instructions 69 / 72 and 97 / 103, 13,000 85 / 76 and
// 103 / 99, 16,000 101 / 86 and 120 / 109.
#define EIGHT_INSTR_ROWS 24000000ull
#define EIGHT_MOST_INSTRS 16000u
#define EIGHT_EDGE_INSTRS 11000u
bool vl_eight_wanted(vl_program *p, uint64_t K)
{
    if (p->group_opt || p->threads_opt) return false;  // the caller asks for the batched kernels
    if (!p->d_ev8 || !p->bank_fast || p->nS > 65535u || !vl_verify_takes(p)) return false;
    if (p->known[VL_KNOWN_SEN] >= FUSED_MANY_ENTRIES || p->known[VL_KNOWN_LS] >= (uint64_t)EXACT_LONG * p->nI) return false;
    const uint64_t wave = 8ull * vl_sm_count(p);
    if (K > wave && (K * p->nI > EIGHT_INSTR_ROWS || p->nI > (6 * K < 7 * wave ? EIGHT_EDGE_INSTRS : EIGHT_MOST_INSTRS))) return false;
    return eight_plan(p, K).NT != 0;
}

// Whether a job may share a launch with jobs of other programs: blocks of 256 threads, two per multiprocessor.
bool vl_eight_shares(vl_program *p, uint64_t K) { return vl_eight_wanted(p, K) && eight_smem(p, 256, E_HALF).total; }

// A job of one program leaves the counts of its rows that collide to k_exact: a row that fails would keep its block busy for longer
// than all the rest takes.  Of more than 2,000 rows of a short program enough blocks are left to go on meanwhile, and k_exact
// costs 4 to 7 us, and more the more rows there are to look through.  Counted by the block / handed over, us, none failing, 10 % and 40 %: 1,000 instructions, 2,368 rows
// 19 / 24, 35 / 38, 49 / 50; 2,000 instructions 24 / 26, 42 / 42, 65 / 55; 3,000 instructions 31 / 33, 62 / 49, 81 / 67; 8,000
// instructions 62 / 62, 119 / 87, 230 / 118; 3,000 instructions, 4,736 rows 59 / 58, 92 / 82, 126 / 122, 8,000 rows 101 / 105,
// 136 / 140, 186 / 189.
#define EIGHT_HAND_ROWS 2000u
#define EIGHT_HAND_INSTRS 2400u

bool vl_eight_hands(vl_program *p, uint64_t rows)
{
    return vl_exact_takes_rows(p, rows) && (rows <= EIGHT_HAND_ROWS || (p->nI >= EIGHT_HAND_INSTRS && rows <= 2ull * p->nI));
}

int vl_eight_run(uint32_t n, vl_program *const *progs, const uint16_t *const *d_cand, const uint64_t *K, const uint64_t *pitch,
                 vl_verdict *const *d_out, cudaStream_t from, cudaStream_t st, bool dict, int slot)
{
    vl_program *p0 = progs[0];
    uint64_t rows = 0;
    uint32_t smem = 0, NT = 256;
    EMany<VL_EIGHT_MANY> many;
    for (uint32_t j = 0; j < n; ++j) {
        vl_program *p = progs[j];
        EParams &e = many.p[j];
        EPlan pl{};
        if (n > 1) {
            pl.NT = 256;
            pl.sm = eight_smem(p, 256, E_HALF);
        } else {
            pl = eight_plan(p, K[j]);
        }
        NT = pl.NT;
        e.f = fused_params(p, dict);
        e.sm = pl.sm;
        e.f.cb = pl.sm.cb;
        e.f.cand = d_cand[j]; e.f.K = K[j]; e.f.pitch = pitch[j]; e.f.out = d_out[j];
        e.nOp8 = dict ? p->nD8 : p->nOp8;
        e.ntiles = (e.nOp8 + NT * 4 - 1) / (NT * 4);
        e.nC = p->nC; e.CW = (p->nC + 31) / 32; e.pf = p->prefetch_tiles;
        e.bank_total = 2 * (p->bank_seg[1] - p->bank_seg[0]) + 3 * (p->bank_seg[2] - p->bank_seg[1]) + 4 * (p->bank_seg[3] - p->bank_seg[2]);
        e.opoff = dict ? p->d_dict_opoff : p->d_opoff; e.first4 = dict ? p->d_dict_first4 : p->d_first4;
        e.ev8 = p->d_ev8; e.cev_off = p->d_cev_off; e.chunk_blk = p->d_chunk_blk; e.short_chunk = p->d_short_chunk;
        e.status = p->d_status + 1; e.test_wait = p->test_wait;
        smem = std::max(smem, pl.sm.total);
        rows = std::max(rows, K[j]);
        const int rc = vl_live_join(p, from, st);
        if (rc != VL_OK) return rc;
    }
    // timing events: the one kernel counts as the table kernel; every handle of a shared launch has the whole launch
    auto mark = [&](int times) {
        for (uint32_t j = 0; j < n; ++j) {
            if (!progs[j]->ktime || std::find(progs, progs + j, progs[j]) != progs + j) continue;
            for (int t = 0; t < times; ++t) kt_mark(progs[j], st);
        }
    };
    mark(1);
    const uint32_t blocks = (uint32_t)((rows + 7) / 8);
    if (n > 1) {
        VL_CUDA(p0, (launch_eight<256, VL_EIGHT_MANY, false>(p0->device, many, dim3(blocks, n), smem, st)));
    } else {
        EMany<1> one;
        one.p[0] = many.p[0];
        if (slot >= 0 && vl_eight_hands(p0, rows)) {
            VlExactArgs &ex = one.p[0].f.ex;
            const int rc = vl_hand_scratch(p0, slot, rows, &ex);
            if (rc != VL_OK) return rc;
            ex.exact_bank = 0;
            if (NT == 512) VL_CUDA(p0, (launch_eight<512, 1, true>(p0->device, one, dim3(blocks), smem, st)));
            else VL_CUDA(p0, (launch_eight<256, 1, true>(p0->device, one, dim3(blocks), smem, st)));
            mark(3);
            const int re = vl_exact_run(p0, ex, d_cand[0], pitch[0], d_out[0], st, dict, true);
            mark(1);
            return re;
        }
        if (NT == 512) VL_CUDA(p0, (launch_eight<512, 1, false>(p0->device, one, dim3(blocks), smem, st)));
        else VL_CUDA(p0, (launch_eight<256, 1, false>(p0->device, one, dim3(blocks), smem, st)));
    }
    mark(4);
    return VL_OK;
}
