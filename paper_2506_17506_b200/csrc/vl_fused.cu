// The whole check of a candidate by one thread block: the verify path of short jobs.
//
// The batched kernels (vl_verify.cu) hand a candidate from kernel to kernel through global memory and want
// thousands of rows; a job of up to a few hundred rows spends its time in their launches and in chains of
// dependent L2 loads.  Here a thread block does everything for its candidate out of shared memory:
//   1. the vreg -> register table T from the first occurrences, with Realizability (file and rules);
//   2. Consistency: every column against T;
//   3. the exact bank tally;
//   4. Safety: one thread per short chunk of instructions toggles the occupancy bits of its chunk's events in
//      a mask of its own (column `tid` of [word][thread]), starting from the block's through-set and what else is
//      occupied on entry (which all threads enter together: it needs no order);
//   5. only if a test found an occupied bit: the exact count of the overlaps in the chunks concerned.
// A vreg at or beyond P takes part in step 4 as if it sat at P: two of them live together then collide, so
// that a chunk is never missed, and step 5 compares the true registers.
#include <algorithm>
#include <mutex>

#include "vl_exact.cuh"

#define EXACT_NT 256
// Coarse items of k_fused's and k_eight's rows: more than four rounds of the blocks become three.  Four / three rounds, us: 8,000
// instructions, 1,184 rows, half of them noise 611 / 526, 32,000 instructions, 749 rows, a tenth 560 / 504; all items, three
// rounds: 24,000 instructions, 999 rows with one fault each 184 / 195, half of them noise 2,464 / 1,416.
#define EXACT_ROUNDS 3
#define EXACT_MOST_ROUNDS 4
#define EXACT_SMEM (224u * 1024)  // shared memory of a block of k_exact, at most
#define EXACT_ROWS 8192           // rows that k_fused and k_eight leave counts of, at most: each block adds up their items

namespace {

inline uint32_t up16(uint32_t x) { return (x + 15u) & ~15u; }

inline FSmem fused_smem(const vl_program *p, uint32_t threads)
{
    const uint32_t Wp = (p->P + p->wmax + 31) / 32;
    FSmem s;
    s.w = up16((p->V + 1) * 2);
    s.th = s.w + up16(p->V + 1);
    s.occ = s.th + (p->use_th ? up16(p->nB * Wp * 4) : 0u);
    const uint32_t counts = (p->P + p->wmax + 2) * 4;  // (of one program block, see exact_counts)
    s.coll = s.occ + up16(std::max(Wp * threads * 4, counts));
    s.cb = p->use_th ? (s.coll - s.occ) / counts : p->nB;
    s.list = s.coll + up16((p->nS + 31) / 32 * 4 + 4);
    s.misc = s.list + up16(p->nS * 8);
    s.total = s.misc + up16(sizeof(FMisc));
    return s;
}

// The jobs of up to N programs in one grid: blockIdx.y is the program.
template <int N>
struct FMany {
    FParams p[N];
};
static_assert(sizeof(FMany<VL_FUSED_MANY>) <= 32764, "kernel arguments");

// BPM: thread blocks per multiprocessor that the registers have to leave room for.  One or two rows per multiprocessor are
// bound by latency (registers for loads in flight), more rows by how many warps there are to switch between: 6,400 rows of
// 64 programs 345 us with two blocks of 256 threads, 281 with three, 274 with four (but spills: one row 20 % slower).
// HAND: candidates with a collision are left to k_exact, which spreads their counts over all multiprocessors.
template <int NTHR, int BPM, int N, bool HAND>
__global__ void __launch_bounds__(NTHR, BPM) k_fused(const __grid_constant__ FMany<N> a)
{
    const FParams &q = a.p[N == 1 ? 0 : blockIdx.y];
    if (N > 1 && blockIdx.x >= q.K) return;
    extern __shared__ __align__(16) unsigned char smem[];
    uint16_t *T = reinterpret_cast<uint16_t *>(smem);                 // [V + 1] register of every vreg
    uint8_t *W = smem + q.sm.w;                                       // [V] width
    uint32_t *s_th = reinterpret_cast<uint32_t *>(smem + q.sm.th);    // [nB][Wp] through-set masks
    uint32_t *occ = reinterpret_cast<uint32_t *>(smem + q.sm.occ);    // [Wp][NTHR] masks; counts in step 5
    uint32_t *coll = reinterpret_cast<uint32_t *>(smem + q.sm.coll);  // short chunks that collided
    uint2 *list = reinterpret_cast<uint2 *>(smem + q.sm.list);        // the same as a list, in step 5
    FMisc *M = reinterpret_cast<FMisc *>(smem + q.sm.misc);
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t k = blockIdx.x;
    const uint16_t *row = q.cand + k * q.pitch;

    if (tid == 0) {
        M->flags = M->bank = M->pairs = M->thcol = M->any = 0;
        M->minop = M->minr = M->mind = 0xFFFFFFFFu;
    }
    pdl_go();
    pdl_wait();  // (the rows, and what liveness computed)
    load_blocks(q, M);
    if (q.use_th)
        for (uint32_t j = tid; j < q.nB * q.Wp; j += NTHR) s_th[j] = 0;
    __syncthreads();

    // Every phase keeps several loads per thread in flight and asks for its first ones before the phase in front of
    // it computes: with one candidate per block the time is a chain of L2 round trips, not work.  Loads past the end
    // of a list take a clamped index and are dropped afterwards: a load under a condition of its own per thread is
    // waited for before the next one is issued.
    constexpr int CU = 3;  // column loads (8 columns each) in flight
    uint4 r_nx[CU], v_nx[CU];
    const uint32_t o_last = q.nO ? (q.nO - 1) & ~7u : 0u;
    auto fetch_columns = [&](uint32_t o0) {
#pragma unroll
        for (int u = 0; u < CU; ++u) {
            const uint32_t o = min(o0 + u * NTHR * 8, o_last);
            r_nx[u] = *reinterpret_cast<const uint4 *>(row + o);
            v_nx[u] = *reinterpret_cast<const uint4 *>(q.vreg16 + o);
        }
    };
    // ---- 1. the table, eight vregs per thread in flight
    for (uint32_t v0 = tid; v0 < q.V; v0 += 8 * NTHR) {
        uint32_t pos[8], vi[8], t[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t v = min(v0 + u * NTHR, q.V - 1);
            pos[u] = q.first_occ[v];
            vi[u] = q.vinfo[v];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            t[u] = row[pos[u] != 0xFFFFFFFFu ? pos[u] : 0u];
            if (pos[u] == 0xFFFFFFFFu) t[u] = 0;
        }
        if (v0 + 8 * NTHR >= q.V) fetch_columns(tid * 8);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t v = v0 + u * NTHR, w = vi[u] & 0xFFu;
            if (v >= q.V) break;
            T[v] = (uint16_t)t[u];
            W[v] = (uint8_t)w;
            if (!(vi[u] & VINFO_DEFINED)) continue;
            bool bad = t[u] + w > q.P;
            if (q.vcons) {
                const uint4 vc = q.vcons[v];
                const uint32_t clo = vc.x & 0xFFFFu, chi = vc.x >> 16, al = vc.y;
                bad = bad || (al > 1 && t[u] != __umulhi(t[u], vc.z) * al) || t[u] < clo || t[u] + w > chi;
                if (!bad && q.rs_prefix) bad = q.rs_prefix[min(t[u] + w, q.P)] != q.rs_prefix[min(t[u], q.P)];
            }
            if (bad) {
                atomicOr(&M->flags, (uint32_t)VL_OUT_OF_RANGE);
                atomicMin(&M->minr, q.first_def_instr[v]);
            }
        }
    }
    if (tid >= q.V) fetch_columns(tid * 8);  // (a thread without a vreg)
    if (tid == 0) T[q.V] = 0;
    __syncthreads();

    // ---- 2. Consistency: 8 columns per load
    constexpr int BU = 6;  // bank list entries in flight
    uint2 id_nx[BU];
    const uint32_t n_ent = q.bank_fast ? q.bank_seg[3] : 0u, ent_last = n_ent ? n_ent - 1 : 0u;
    auto fetch_bank = [&](uint32_t e0) {
#pragma unroll
        for (int u = 0; u < BU; ++u) id_nx[u] = q.bank_list[min(e0 + u * NTHR, ent_last)];
    };
    for (uint32_t o0 = tid * 8; o0 < q.nO; o0 += CU * NTHR * 8) {
        uint4 r4[CU], v4[CU];
#pragma unroll
        for (int u = 0; u < CU; ++u) { r4[u] = r_nx[u]; v4[u] = v_nx[u]; }
        if (o0 + CU * NTHR * 8 < q.nO) fetch_columns(o0 + CU * NTHR * 8);
        else fetch_bank(tid);
#pragma unroll
        for (int u = 0; u < CU; ++u) {
            const uint32_t o = o0 + u * NTHR * 8;
            if (o >= q.nO) break;
            const uint32_t r[4] = {r4[u].x, r4[u].y, r4[u].z, r4[u].w}, v[4] = {v4[u].x, v4[u].y, v4[u].z, v4[u].w};
            uint32_t d[4], any = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                d[j] = r[j] ^ ((uint32_t)T[v[j] & 0xFFFFu] | ((uint32_t)T[v[j] >> 16] << 16));
                any |= d[j];
            }
            if (any) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (((j & 1) ? d[j >> 1] >> 16 : d[j >> 1] & 0xFFFFu) && o + j < q.nO) {
                        atomicOr(&M->flags, (uint32_t)VL_INCONSISTENT);
                        atomicMin(&M->minop, o + j);
                    }
            }
        }
    }
    if (tid * 8 >= q.nO) fetch_bank(tid);  // (a thread without a column)

    // ---- 3. bank tally
    {
        uint32_t n = 0;
        for (uint32_t e0 = tid; e0 < n_ent; e0 += BU * NTHR) {
            uint2 id[BU];
#pragma unroll
            for (int u = 0; u < BU; ++u) id[u] = id_nx[u];
            fetch_bank(e0 + BU * NTHR);
#pragma unroll
            for (int u = 0; u < BU; ++u) {
                const uint32_t e = e0 + u * NTHR;
                if (e >= n_ent) break;
                n += bank_entry(id[u], e < q.bank_seg[1] ? 2u : (e < q.bank_seg[2] ? 3u : 4u), T, q.B - 1);
            }
        }
        if (!q.bank_fast) {
            for (uint32_t i = tid; i < q.nI; i += NTHR) n += bank_instr(q, T, i);
        }
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0 && n) atomicAdd(&M->bank, n);
    }

    // ---- 4. Safety
    if (q.use_th) {
        const uint32_t n_th = M->th_off[q.nB];
        for (uint32_t e = tid; e < n_th; e += NTHR) {
            const uint32_t x = q.th[e];
            uint32_t b = 0;
            while (b + 1 < q.nB && M->th_off[b + 1] <= e) ++b;
            uint32_t pos = min((uint32_t)T[x & 0xFFFFu], q.P), left = x >> 16;
            bool hit = false;
            while (left) {
                const uint32_t s2 = pos & 31, n = min(left, 32 - s2);
                const uint32_t m = (0xFFFFFFFFu >> (32 - n)) << s2;
                hit |= (atomicOr(&s_th[b * q.Wp + (pos >> 5)], m) & m) != 0;
                pos += n;
                left -= n;
            }
            if (hit) atomicOr(&M->thcol, 1u << b);  // through-sets are used only if nB <= 32
        }
        __syncthreads();
    }
    const uint32_t nSr = (q.nS + 31u) & ~31u;
    for (uint32_t s0 = 0; s0 < nSr; s0 += NTHR) {  // (a warp takes a whole group of 32 short chunks)
        const uint32_t s = s0 + tid;
        const bool mine = s < nSr;
        const uint32_t st0 = mine ? q.sev_off[s >> 5] : 0u, steps = mine ? q.sev_off[(s >> 5) + 1] - st0 : 0u;
        const uint32_t *ev = q.sev + (size_t)st0 * 32 + lane;
        const uint32_t step_last = steps ? steps - 1 : 0u;
        constexpr int EU = 8;  // events in flight: loaded ahead, and applied
        uint32_t nx[EU];
#pragma unroll
        for (int u = 0; u < EU; ++u) nx[u] = ev[(size_t)min((uint32_t)u, step_last) * 32];
        uint32_t en[4];
        const uint32_t e_hi = q.sen_off[min(q.nS, s0 + NTHR)], e_lo = q.sen_off[s0], e_end = max(e_hi, 1u) - 1;
#pragma unroll
        for (int u = 0; u < 4; ++u) en[u] = q.sen[min(e_lo + tid + u * NTHR, e_end)];
        const uint32_t b = s < q.nS && q.use_th ? q.short_blk[s] : 0u;
        for (uint32_t wd = 0; wd < q.Wp; ++wd) occ[wd * NTHR + tid] = q.use_th ? s_th[b * q.Wp + wd] : 0u;
        if (mine && lane == 0) coll[s >> 5] = 0;
        __syncthreads();
        for (uint32_t e0 = e_lo + tid; e0 < e_hi; e0 += 4 * NTHR) {
            uint32_t x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                x[u] = en[u];
                en[u] = q.sen[min(e0 + (4 + u) * NTHR, e_end)];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e0 + u * NTHR >= e_hi) break;
                const uint32_t v = x[u] & 0xFFFFu, col = ((x[u] >> 16) - s0) & 0xFFFFu;
                uint32_t pos = min((uint32_t)T[v], q.P), left = W[v];
                bool hit = false;
                while (left) {
                    const uint32_t s2 = pos & 31, n = min(left, 32 - s2);
                    const uint32_t m = (0xFFFFFFFFu >> (32 - n)) << s2;
                    hit |= (atomicOr(&occ[(pos >> 5) * NTHR + col], m) & m) != 0;
                    pos += n;
                    left -= n;
                }
                if (hit) { atomicOr(&coll[(s0 + col) >> 5], 1u << (col & 31)); M->any = 1; }
            }
        }
        __syncthreads();
        uint32_t viol = 0;
        for (uint32_t e0 = 0; e0 < steps; e0 += EU) {
            uint32_t x[EU], t[EU], old[EU];
            uint32_t far = 0;  // some range of the batch reaches into the next word
#pragma unroll
            for (int u = 0; u < EU; ++u) {
                x[u] = e0 + u < steps ? nx[u] : 0u;
                t[u] = min((uint32_t)T[x[u] & 0xFFFFu], q.P);
                far |= (t[u] & 31) + ((x[u] >> 16) & 0xFFu) > 32 ? 1u : 0u;
                nx[u] = ev[(size_t)min(e0 + EU + u, step_last) * 32];
            }
            // toggling returns the old word: occupied and released are both a toggle as long as no collision
            // has been seen (after one, the chunk is counted exactly anyway)
            if (!far) {
#pragma unroll
                for (int u = 0; u < EU; ++u) {
                    const uint32_t w = (x[u] >> 16) & 0xFFu, m = w ? (0xFFFFFFFFu >> (32 - w)) << (t[u] & 31) : 0u;
                    old[u] = atomicXor(&occ[(t[u] >> 5) * NTHR + tid], (x[u] >> 25) & 1u ? m : 0u);
                    t[u] = (x[u] >> 24) & 1u ? m : 0u;
                }
#pragma unroll
                for (int u = 0; u < EU; ++u) viol |= old[u] & t[u];
            } else {
#pragma unroll 1
                for (int u = 0; u < EU; ++u) {
                    uint32_t xu = x[0], pos = t[0];
#pragma unroll
                    for (int j = 1; j < EU; ++j)
                        if (j == u) { xu = x[j]; pos = t[j]; }
                    const uint32_t tog = 0u - ((xu >> 25) & 1u), test = 0u - ((xu >> 24) & 1u);
                    uint32_t left = (xu >> 16) & 0xFFu;
                    while (left) {
                        const uint32_t s2 = pos & 31, n = min(left, 32 - s2);
                        const uint32_t m = (0xFFFFFFFFu >> (32 - n)) << s2;
                        viol |= atomicXor(&occ[(pos >> 5) * NTHR + tid], m & tog) & m & test;
                        pos += n;
                        left -= n;
                    }
                }
            }
        }
        const uint32_t hits = __ballot_sync(0xffffffffu, viol != 0);
        if (mine && lane == 0 && hits) {
            atomicOr(&coll[s >> 5], hits);
            M->any = 1;
        }
        __syncthreads();
    }
    __syncthreads();

    // ---- 5. exact counts where something collided
    const bool collided = M->any | M->thcol;
    if (!HAND && collided) exact_counts<NTHR, false>(q, T, W, occ, coll, list, M, 0, 1, row);

    // ---- the verdict
    if (warp == 0) {
        uint32_t first = min(M->minr, M->mind);
        const uint32_t o = M->minop;
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
        if (HAND && collided) {
            uint32_t chunks = M->thcol ? q.ex.nC / 8 : 0u;  // (the sources in the through-set)
            for (uint32_t w = 0; w < q.ex.AW; ++w) {
                const uint32_t c = w * 32 + lane;
                bool hit = false;
                if (c < q.ex.nC)
                    for (uint32_t s = q.ex.chunk_short_off[c]; s < q.ex.chunk_short_off[c + 1]; ++s) hit |= (coll[s >> 5] >> (s & 31)) & 1u;
                const uint32_t bits = __ballot_sync(0xffffffffu, hit);
                if (lane == 0) q.ex.anom[k * q.ex.AW + w] = bits;
                chunks += __popc(bits);
            }
            if (lane < 4) q.ex.racc[k * 4 + lane] = 0;
            if (lane == 0) {
                uint32_t *cs = q.ex.cstate + k * 8;
                cs[CS_FLAGS] = M->flags; cs[CS_FIRST] = first; cs[CS_BANK] = M->bank;
                cs[CS_WALK] = M->any ? WALK_ANOM : 0u; cs[CS_THCOL] = M->thcol;
                q.ex.items[k] = exact_parts(chunks, EXACT_PART_CHUNKS) | exact_parts(chunks, EXACT_FINE_CHUNKS) << 16;
            }
        } else if (lane == 0) {
            if (HAND) q.ex.items[k] = 0;
            const uint32_t flags = M->flags | (M->pairs ? (uint32_t)VL_INTERFERENCE : 0u);
            vl_verdict vd;
            vd.flags = flags ? flags : (uint32_t)VL_PASS;
            vd.first_violation_instr = first == 0xFFFFFFFFu ? -1 : (int32_t)first;
            vd.conflict_pairs = M->pairs;
            vd.bank_conflicts = M->bank;
            q.out[k] = vd;
        }
    }
}

// Candidates of the batched kernels that need an exact count (their walk collided, several of their vregs lie outside the
// file, or the program has no fast bank tally), listed in work as items of one or several parts per candidate; a thread
// block takes an item.  Consistency and Realizability are in cstate; a chunk of the walk that collided marks all of its
// short chunks.  GLOBAL: the block's arrays lie in a slice of global memory (programs that do not fit a multiprocessor).
// ROWS: the candidates are the rows of k_fused or k_eight, which left the number of items of each; every block adds them up
// for itself (a list with its counts would have to be cleared in front of every call: 3.3 us of 26 for 200 rows of 8,000
// instructions by a memset; reset by the last block, it is left as it is by a call whose second launch fails).
template <bool GLOBAL, bool ROWS, bool LONG>
__global__ void __launch_bounds__(EXACT_NT, 2) k_exact(const __grid_constant__ FParams q)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ FMisc misc;
    FMisc *M = &misc;
    unsigned char *base = GLOBAL ? q.ex.scratch + (size_t)blockIdx.x * q.sm.total : smem;
    uint16_t *T = reinterpret_cast<uint16_t *>(base);
    uint8_t *W = base + q.sm.w;
    uint32_t *occ = reinterpret_cast<uint32_t *>(base + q.sm.occ), *coll = reinterpret_cast<uint32_t *>(base + q.sm.coll);
    uint2 *list = reinterpret_cast<uint2 *>(base + q.sm.list);
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    pdl_wait();
    uint32_t n_items;
    const uint32_t *items = nullptr;
    uint32_t *first = reinterpret_cast<uint32_t *>(base + q.sm.total);  // ROWS: [rows + 1] first item of every row
    if (ROWS) {
        using u64 = unsigned long long;
        __shared__ u64 s_sum[EXACT_NT / 32];
        constexpr uint32_t U = 8;
        bool any = false;
        for (uint32_t k0 = tid; k0 < q.ex.rows; k0 += U * EXACT_NT) {
            uint32_t x[U];
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) x[u] = q.ex.items[min(k0 + u * EXACT_NT, q.ex.rows - 1)];
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                if (k0 + u * EXACT_NT < q.ex.rows) first[k0 + u * EXACT_NT] = x[u];
                any |= x[u] != 0;
            }
        }
        if (!__syncthreads_or(any)) return;
        // (an odd number of rows per thread: their places begin in different banks)
        const uint32_t per = (q.ex.rows + EXACT_NT - 1) / EXACT_NT | 1u, k0 = tid * per, k1 = min(k0 + per, q.ex.rows);
        auto scan = [&](u64 n, u64 &all) {  // of the threads in front of this one; of all
            u64 inc = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const u64 y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= (uint32_t)d) inc += y;
            }
            __syncthreads();
            if (lane == 31) s_sum[tid >> 5] = inc;
            __syncthreads();
            u64 before = inc - n;
            all = 0;
#pragma unroll
            for (uint32_t w = 0; w < EXACT_NT / 32; ++w) {
                if (w < tid >> 5) before += s_sum[w];
                all += s_sum[w];
            }
            return before;
        };
        u64 n = 0, all;  // coarse items, fine items << 32
        for (uint32_t k = k0; k < k1; ++k) n += (first[k] & 0xFFFFu) | (u64)(first[k] >> 16) << 32;
        u64 before = scan(n, all);
        // Fine items if each has a thread block; else coarse ones, and no more of them than a few rounds of the blocks take: an item
        // fetches its part of the row anew (15 to 20 us) and counts it.
        const uint32_t coarse = (uint32_t)all, most = EXACT_ROUNDS * gridDim.x;
        const bool fine = (uint32_t)(all >> 32) <= q.ex.fine_items, fewer = !fine && coarse > EXACT_MOST_ROUNDS * gridDim.x;
        auto of_row = [&](uint32_t x) {
            if (fine) return x >> 16;
            x &= 0xFFFFu;
            return fewer && x ? max(1u, x * most / coarse) : x;
        };
        if (fewer) {
            n = 0;
            for (uint32_t k = k0; k < k1; ++k) n += of_row(first[k]);
            before = scan(n, all);
        }
        n_items = (uint32_t)(fine ? all >> 32 : all);
        uint32_t at = (uint32_t)(fine ? before >> 32 : before);
        for (uint32_t k = k0; k < k1; ++k) {
            const uint32_t x = of_row(first[k]);
            first[k] = at;
            at += x;
        }
        if (tid == 0) first[q.ex.rows] = n_items;
        __syncthreads();
    } else {
        const bool fine = q.ex.work[1] <= q.ex.fine_items;
        n_items = q.ex.work[fine ? 1 : 0];
        items = q.ex.work + EXACT_HDR + (fine ? 0 : 2 * EXACT_FINE_ITEMS);
    }
    for (uint32_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        uint64_t k;
        uint32_t part, parts;
        if (ROWS) {
            uint32_t lo = 0, hi = q.ex.rows;  // first[lo] <= it < first[hi]
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (first[mid] <= it) lo = mid; else hi = mid;
            }
            k = lo;
            part = it - first[lo];
            parts = first[lo + 1] - first[lo];
        } else {
            k = items[2 * it];
            part = items[2 * it + 1] & 0xFFu;
            parts = items[2 * it + 1] >> 8;
        }
        const uint16_t *row = q.cand + k * q.pitch;
        const uint32_t *cs = q.ex.cstate + k * 8;
        const uint32_t walk = cs[CS_WALK], thcol = cs[CS_THCOL];
        const bool full = walk & WALK_FULL;
        __syncthreads();
        if (tid == 0) {
            M->bank = M->pairs = M->dups = 0;
            M->thcol = full ? 0u : thcol;  // (with every chunk counted in full, nothing is left of the through-sets)
            M->mind = 0xFFFFFFFFu;
        }
        load_blocks(q, M);
        const bool count = (walk | thcol) != 0;
        if (count)
            for (uint32_t s = tid; s < ((q.nS + 31u) & ~31u); s += EXACT_NT) {
                const uint32_t c = q.ex.short_chunk[min(s, q.nS - 1)];
                const bool hit = s < q.nS && (full || ((q.ex.anom[k * q.ex.AW + (c >> 5)] >> (c & 31)) & 1u));
                const uint32_t bits = __ballot_sync(0xffffffffu, hit);
                if (lane == 0) coll[s >> 5] = bits;
            }
        __syncthreads();
        if (count) exact_counts<EXACT_NT, true, LONG>(q, T, W, occ, coll, list, M, part, parts, row);
        __syncthreads();
        if (ROWS || q.bank_fast) {
            if (tid == 0) M->bank = (part == 0 ? cs[CS_BANK] : 0u) - (ROWS && q.ex.exact_bank ? 0u : M->dups);
        } else {  // the general tally: the whole table, this part's instructions
            for (uint32_t v0 = tid; v0 < q.V; v0 += 8 * EXACT_NT) {
                uint32_t pos[8], t[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) pos[u] = q.first_occ[min(v0 + u * EXACT_NT, q.V - 1)];
#pragma unroll
                for (int u = 0; u < 8; ++u) t[u] = row[pos[u] != 0xFFFFFFFFu ? pos[u] : 0u];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (v0 + u * EXACT_NT < q.V) T[v0 + u * EXACT_NT] = pos[u] != 0xFFFFFFFFu ? (uint16_t)t[u] : (uint16_t)0;
            }
            __syncthreads();
            uint32_t n = bank_instrs(q, T, (uint32_t)((uint64_t)q.nI * part / parts), (uint32_t)((uint64_t)q.nI * (part + 1) / parts));
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0 && n) atomicAdd(&M->bank, n);
        }
        __syncthreads();
        if (tid == 0) {
            uint32_t pairs = M->pairs, mind = M->mind, bank = M->bank;
            bool last = true;
            if (parts > 1) {  // accumulators start at 0: the complement of the lowest instruction
                uint32_t *acc = q.ex.racc + k * 4;
                if (pairs) { atomicAdd(&acc[0], pairs); atomicMax(&acc[1], ~mind); }
                if (bank) atomicAdd(&acc[2], bank);
                __threadfence();
                last = atomicAdd(&acc[3], 1u) == parts - 1;
                if (last) {
                    __threadfence();
                    pairs = atomicAdd(&acc[0], 0u);
                    mind = ~atomicMax(&acc[1], 0u);
                    bank = atomicAdd(&acc[2], 0u);
                }
            }
            if (last) {
                const uint32_t flags = cs[CS_FLAGS] | (pairs ? (uint32_t)VL_INTERFERENCE : 0u), first = min(cs[CS_FIRST], mind);
                vl_verdict vd;
                vd.flags = flags ? flags : (uint32_t)VL_PASS;
                vd.first_violation_instr = first == 0xFFFFFFFFu ? -1 : (int32_t)first;
                vd.conflict_pairs = pairs;
                vd.bank_conflicts = bank;
                q.out[k] = vd;
            }
        }
    }
}

// How a job of K rows runs: threads per block (0: the program does not fit the kernel), blocks per multiprocessor.  Up to
// one row per multiprocessor a block takes a whole one; for more rows two or three blocks share one, where their masks let
// them (a program of 8,000 instructions: 16.6 us for 148 rows, 38 us for 300).
struct FPlan {
    uint32_t threads, bpm;
};
FPlan fused_plan(vl_program *p, uint64_t K)
{
    const uint32_t cap = 227 * 1024;
    const uint64_t sms = (uint64_t)vl_sm_count(p);
    if (p->nS > 65535u) return {0, 0};
    const uint32_t half = fused_smem(p, 256).total, full = fused_smem(p, 512).total;
    if (K > 2 * sms && 3 * (half + 1024) <= cap) return {256, 3};
    if (K > sms && 2 * (half + 1024) <= cap) return {256, 2};
    return {full <= cap ? 512u : (half <= cap ? 256u : 0u), 1};
}

}  // namespace

// Jobs whose rows the device holds at a time: 10 us against 45 for 100 rows of a program of 2,000 instructions, 40
// against 81 for 148 rows of one of 8,000 (14 against 66 when no row fails), 54 against 146 for one of 32,000.  Beyond
// that the batched kernels, which read the program's tables for 8 or 64 rows at a time, win as soon as the rounds of
// this kernel (about 3 us and 3.5 ns per instruction) take longer than their launches: 600 rows of 2,000 instructions 31
// against 42 us, 1,000 rows 41 against 42; 3,000 rows of 64 instructions 40 against 68, 10,000 rows 124 against 79.
// A program whose short chunks begin with many vregs occupied is something else: a row enters them all by itself and counts
// its collisions in lists as long, which the batched kernels spread over the multiprocessors.  3,500 instructions with 500
// vregs live everywhere, rows that collide everywhere: 1 row 101 us against 410, 100 rows 320 against 416, 148 rows 424
// against 418, 300 rows 690 against 1,211; 24,300 instructions with 300 such vregs: 1 row 0.56 ms against 13, 127 rows 29.8
// against 13, 148 rows 34.7 against 13.  (The line, 49,152 entries: one row of 860 instructions with 200 vregs, 22,000 entries,
// takes 60 us here and 65 there, of 1,620 with 300, 60,000 entries, 115 and 74; of 800 with 600 of which 200 read 60 vregs each,
// 37,000 entries and no fast bank tally, 192 and 423.  Programs whose values live shortly have below 10,000.)
#define FUSED_FEW_ROWS 128u
// 100 rows that collide everywhere, a warp per instruction against a thread: lists of 2,330 entries on average 5,916 us against
// 8,602, of 1,013 1,441 against 1,261, of 557 640 against 454.
static bool long_lists(const vl_program *p) { return p->known[VL_KNOWN_LS] >= (uint64_t)EXACT_LONG * p->nI; }

bool vl_fused_wanted(vl_program *p, uint64_t K, bool alone)
{
    if (p->group_opt || p->threads_opt || p->test_wait) return false;  // the caller asks for the batched kernels
    if (!vl_verify_takes(p)) return false;                             // (refused, however few the rows)
    if (p->known[VL_KNOWN_SEN] >= FUSED_MANY_ENTRIES && (K < FUSED_FEW_ROWS || K > (uint64_t)vl_sm_count(p) || long_lists(p))) return false;
    const FPlan pl = fused_plan(p, K);
    if (!pl.threads) return false;
    const uint64_t resident = (uint64_t)pl.bpm * vl_sm_count(p);
    const uint64_t rounds = (K + resident - 1) / resident;
    // Where k_eight takes the job it wins sooner: 1,000 instructions, 1,184 rows 32 us against 34 there, 1,600 rows 40 against 34;
    // 2,000 instructions, 600 rows 29 against 36, 1,000 rows 47 against 38; 4,000 instructions, 400 rows 36 against 40, 600 rows 61
    // against 39.
    return rounds <= 1 || rounds * (6000 + 7ull * p->nI) <= (alone && vl_eight_wanted(p, K) ? 42000u : 72000u);
}

// Programs of at least that many instructions whose rows share multiprocessors hand the exact counts to k_exact: a row that
// fails used to keep its few warps busy for longer than all the rest took, now every multiprocessor shares in it.  300 rows
// of 8,000 instructions 45 us against 88 with 10 % of the rows failing, of 11,317 instructions 62 against 90; with none
// failing the second launch costs 1 us (32.9, 46.0).  Of 5,000 instructions it gains nothing (46.4 against 43.1, 48.2 against
// 48.5 with 30 % failing), nor do rows that have a multiprocessor to themselves (50 rows of 11,317 instructions 22 us).
#define FUSED_HAND_INSTRS 7000u

int vl_hand_scratch(vl_program *p, int slot, uint64_t rows, VlExactArgs *ex)
{
    ex->rows = (uint32_t)rows;
    ex->exact_bank = 1;
    vl_program::VScratch &v = p->fs[slot];
    const uint64_t aw = (p->nC + 31) / 32;
    if (v.rows < rows || v.aw != aw) {
        VL_CUDA(p, cudaFree(v.block));
        v = vl_program::VScratch{};
        rows = std::max<uint64_t>(rows, 3ull * vl_sm_count(p));
        VL_CUDA(p, cudaMalloc(&v.block, rows * (8 + 4 + 1 + aw) * 4));
        v.cstate = static_cast<uint32_t *>(v.block); v.racc = v.cstate + rows * 8; v.work = v.racc + rows * 4; v.anom = v.work + rows;
        v.rows = rows; v.aw = aw;
    }
    ex->cstate = v.cstate; ex->racc = v.racc; ex->items = v.work; ex->anom = v.anom;
    ex->AW = (uint32_t)aw; ex->nC = p->nC;
    ex->short_chunk = p->d_short_chunk; ex->chunk_short_off = p->d_chunk_short_off;
    ex->fine_items = std::min<uint32_t>(vl_exact_blocks(p), EXACT_FINE_ITEMS);
    return VL_OK;
}

// Up to VL_FUSED_MANY jobs in one launch on st.
int vl_fused_run(uint32_t n, vl_program *const *progs, const uint16_t *const *d_cand, const uint64_t *K, const uint64_t *pitch,
                 vl_verdict *const *d_out, cudaStream_t from, cudaStream_t st, bool dict, int slot)
{
    vl_program *p0 = progs[0];
    static std::mutex mtx;
    static bool done[64];
    if (p0->device >= 0 && p0->device < 64) {
        std::lock_guard<std::mutex> lock(mtx);
        if (!done[p0->device]) {
            const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
            VL_CUDA(p0, cudaFuncSetAttribute(k_fused<512, 1, 1, false>, at, 227 * 1024));
            VL_CUDA(p0, cudaFuncSetAttribute(k_fused<256, 2, 1, false>, at, 227 * 1024));
            VL_CUDA(p0, cudaFuncSetAttribute(k_fused<256, 3, 1, false>, at, 227 * 1024));
            VL_CUDA(p0, cudaFuncSetAttribute(k_fused<256, 3, VL_FUSED_MANY, false>, at, 227 * 1024));
            VL_CUDA(p0, cudaFuncSetAttribute(k_fused<256, 2, 1, true>, at, 227 * 1024));
            VL_CUDA(p0, cudaFuncSetAttribute(k_fused<256, 3, 1, true>, at, 227 * 1024));
            done[p0->device] = true;
        }
    }
    uint64_t rows = 0;
    uint32_t smem = 0;
    const FPlan pl = n > 1 ? FPlan{256, 3} : fused_plan(p0, K[0]);
    FMany<VL_FUSED_MANY> many;
    for (uint32_t j = 0; j < n; ++j) {
        vl_program *p = progs[j];
        FParams &q = many.p[j];
        q = fused_params(p, dict);
        q.sm = fused_smem(p, pl.threads);
        q.cb = q.sm.cb;
        smem = std::max(smem, q.sm.total);
        q.cand = d_cand[j]; q.K = K[j]; q.pitch = pitch[j]; q.out = d_out[j];
        rows = std::max(rows, K[j]);
        const int rc = vl_live_join(p, from, st);
        if (rc != VL_OK) return rc;
    }
    // timing events: a job's one kernel counts as the table kernel, what it hands over as the exact counts; every handle of a
    // shared launch has the whole launch
    auto mark = [&](int times) {
        for (uint32_t j = 0; j < n; ++j) {
            if (!progs[j]->ktime || std::find(progs, progs + j, progs[j]) != progs + j) continue;
            for (int t = 0; t < times; ++t) kt_mark(progs[j], st);
        }
    };
    mark(1);
    if (n > 1) {
        VL_CUDA(p0, launch_overlap(k_fused<256, 3, VL_FUSED_MANY, false>, dim3((uint32_t)rows, n), 256, smem, st, true, many));
    } else {
        FMany<1> one;
        one.p[0] = many.p[0];
        const dim3 grid((uint32_t)rows);
        if (slot >= 0 && pl.bpm > 1 && p0->nI >= FUSED_HAND_INSTRS && vl_exact_takes_rows(p0, rows)) {
            VlExactArgs &ex = one.p[0].ex;
            const int rc = vl_hand_scratch(p0, slot, rows, &ex);
            if (rc != VL_OK) return rc;
            VL_CUDA(p0, pl.bpm == 3 ? launch_overlap(k_fused<256, 3, 1, true>, grid, 256, smem, st, true, one)
                                    : launch_overlap(k_fused<256, 2, 1, true>, grid, 256, smem, st, true, one));
            mark(3);
            const int re = vl_exact_run(p0, ex, d_cand[0], pitch[0], d_out[0], st, dict, true);
            mark(1);
            return re;
        }
        if (pl.threads == 512) VL_CUDA(p0, launch_overlap(k_fused<512, 1, 1, false>, grid, 512, smem, st, true, one));
        else if (pl.bpm == 3) VL_CUDA(p0, launch_overlap(k_fused<256, 3, 1, false>, grid, 256, smem, st, true, one));
        else VL_CUDA(p0, launch_overlap(k_fused<256, 2, 1, false>, grid, 256, smem, st, true, one));
    }
    mark(4);
    return VL_OK;
}

// Whether a job may share a launch with jobs of other programs: blocks of 256 threads, small enough that several
// share a multiprocessor whatever the others need.
bool vl_fused_shares(vl_program *p, uint64_t K)
{
    return vl_fused_wanted(p, K, false) && fused_smem(p, 256).total <= 48 * 1024;
}

// Shared memory of a block of k_exact; beyond what a multiprocessor has, its arrays take global memory.
static FSmem exact_smem(const vl_program *p)
{
    FSmem s{};
    s.w = up16((p->V + 1) * 2);
    s.occ = s.w + up16(p->V + 1);
    const uint32_t counts = (p->P + p->wmax + 2) * 4;
    s.cb = p->use_th ? std::max(1u, std::min(p->nB, 48u * 1024u / counts)) : p->nB;
    s.coll = s.occ + (p->use_th ? up16(s.cb * counts) : 0u);
    s.list = s.coll + up16((p->nS + 31) / 32 * 4 + 4);
    s.total = s.list + up16(p->nS * 8) + p->nC * 16;
    return s;
}

uint32_t vl_exact_blocks(vl_program *p)
{
    const uint32_t bytes = exact_smem(p).total;
    return (uint32_t)vl_sm_count(p) * (bytes <= 110 * 1024 ? 2u : 1u);
}

uint64_t vl_exact_scratch(vl_program *p)
{
    const uint64_t bytes = exact_smem(p).total;
    return bytes <= EXACT_SMEM ? 0 : bytes * vl_exact_blocks(p);
}

bool vl_exact_takes_rows(vl_program *p, uint64_t rows)
{
    return rows <= EXACT_ROWS && exact_smem(p).total + (rows + 1) * 4 <= EXACT_SMEM;
}

int vl_exact_run(vl_program *p, const VlExactArgs &ex, const uint16_t *d_cand, uint64_t pitch, vl_verdict *d_out, cudaStream_t st,
                 bool dict, bool overlap)
{
    static std::mutex mtx;
    static bool done[64];
    if (p->device >= 0 && p->device < 64) {
        std::lock_guard<std::mutex> lock(mtx);
        if (!done[p->device]) {
            VL_CUDA(p, cudaFuncSetAttribute(k_exact<false, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, EXACT_SMEM));
            VL_CUDA(p, cudaFuncSetAttribute(k_exact<false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, EXACT_SMEM));
            VL_CUDA(p, cudaFuncSetAttribute(k_exact<false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, EXACT_SMEM));
            done[p->device] = true;
        }
    }
    FParams q = fused_params(p, dict);
    q.sm = exact_smem(p);
    q.cb = q.sm.cb;
    q.ex = ex;
    q.cand = d_cand; q.pitch = pitch; q.out = d_out;
    const uint32_t grid = vl_exact_blocks(p);
    if (ex.rows) VL_CUDA(p, launch_overlap(k_exact<false, true, false>, grid, EXACT_NT, q.sm.total + (ex.rows + 1) * 4, st, overlap, q));
    else if (ex.scratch) VL_CUDA(p, launch_overlap(k_exact<true, false, false>, grid, EXACT_NT, 0, st, overlap, q));
    else if (long_lists(p)) VL_CUDA(p, launch_overlap(k_exact<false, false, true>, grid, EXACT_NT, q.sm.total, st, overlap, q));
    else VL_CUDA(p, launch_overlap(k_exact<false, false, false>, grid, EXACT_NT, q.sm.total, st, overlap, q));
    return VL_OK;
}
