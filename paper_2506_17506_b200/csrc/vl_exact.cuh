// Exact counts of a candidate's overlaps and bank conflicts, shared by the kernels that check candidates out of shared memory.
#pragma once
#include "vl_internal.cuh"

namespace {

struct FMisc {
    uint32_t flags, minop, minr, bank, pairs, mind, thcol, any;
    uint32_t n_list, n_chunks, dups;
    uint32_t blk_i[33], el_n[32], el_o[32];  // first instruction; definitions without an event: how many, first of the list
    uint32_t th_off[33];  // (through-sets are used only by programs of at most 32 blocks)
};

// Where the parts of a block's shared memory start (bytes), and how much there is.
struct FSmem {
    uint32_t w, th, occ, coll, list, misc, total;
    uint32_t cb;  // program blocks whose register counts fit the masks' place
};

struct FParams {
    uint32_t nI, V, nO, P, B, nB, nS, Wp, R, Wv, wmax, short_len, cb;
    int bank_fast, use_th;
    FSmem sm;
    const uint32_t *first_occ, *vinfo, *first_def_instr, *op_off, *op_vreg, *entry_instr, *blk_off;
    const uint16_t *vreg16;
    const uint8_t *opflags;
    const uint8_t *ndefs;
    const uint4 *vcons;
    const uint16_t *rs_prefix;
    const uint2 *bank_list;
    uint32_t bank_seg[4];
    // liveness results
    const uint32_t *th_off, *th, *blk_th, *sev_off, *sev, *sen_off, *sen, *short_blk, *short_i0, *blk_short_off;
    const uint32_t *ls, *el_count;
    const uint4 *el, *irec;
    const uint16_t *cand;
    uint64_t K, pitch;
    vl_verdict *out;
    VlExactArgs ex;  // (k_exact)
};

__device__ __forceinline__ bool overlap(uint32_t a, uint32_t wa, uint32_t b, uint32_t wb) { return a < b + wb && b < a + wa; }

// Sources of one list entry that cost a cycle: the register is new among the entry's sources, its bank is not.
template <int N>
__device__ __forceinline__ uint32_t bank_extra(const uint32_t (&x)[4], uint32_t bmask)
{
    uint32_t n = 0;
#pragma unroll
    for (int a = 1; a < N; ++a) {
        bool value = false, bank = false;
#pragma unroll
        for (int b = 0; b < a; ++b) {
            value |= x[b] == x[a];
            bank |= ((x[b] ^ x[a]) & bmask) == 0;
        }
        n += !value && bank;
    }
    return n;
}
// An entry with n = 2, 3 or 4 distinct source vregs.
__device__ __forceinline__ uint32_t bank_entry(const uint2 &id, uint32_t n, const uint16_t *T, uint32_t bmask)
{
    const uint32_t x[4] = {T[id.x & 0xFFFFu], T[id.x >> 16], T[id.y & 0xFFFFu], T[id.y >> 16]};
    return n == 2 ? bank_extra<2>(x, bmask) : (n == 3 ? bank_extra<3>(x, bmask) : bank_extra<4>(x, bmask));
}

// The same for instruction i of a program without a list (banks not 1, 2 or 4, or more than four distinct sources).
__device__ __forceinline__ uint32_t bank_instr(const FParams &q, const uint16_t *T, uint32_t i)
{
    uint32_t n = 0;
    const uint32_t u0 = q.op_off[i] + q.ndefs[i], u1 = q.op_off[i + 1];
    for (uint32_t a = u0 + 1; a < u1; ++a) {
        const uint32_t xa = T[q.op_vreg[a]];
        bool value = false, bank = false;
        for (uint32_t b = u0; b < a; ++b) {
            const uint32_t xb = T[q.op_vreg[b]];
            value |= xb == xa;
            bank |= xb % q.B == xa % q.B;
        }
        n += !value && bank;
    }
    return n;
}

// The same for instructions [i0, i1), counted by a whole block: four instructions of a thread in flight, from their records;
// an instruction of more than four reads by a warp, a lane per read.  Returns this thread's share.
__device__ __noinline__ uint32_t bank_instrs(const FParams &q, const uint16_t *T, uint32_t i0, uint32_t i1)
{
    constexpr uint32_t U = 4;
    const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1u;
    uint32_t n = 0;
    for (uint32_t base = i0 + (threadIdx.x & ~31u); base < i1; base += U * blockDim.x) {  // (the same for a whole warp)
        uint4 rec[U];
        uint32_t rd[U][4];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) rec[u] = q.irec[min(base + lane + u * blockDim.x, q.nI - 1)];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const uint32_t nr = (rec[u].y >> 24) & 127u, o = rec[u].w + ((rec[u].y >> 16) & 0xFFu);
#pragma unroll
            for (uint32_t r = 0; r < 4; ++r) rd[u][r] = q.op_vreg[nr ? o + min(r, nr - 1) : 0u];  // (missing reads repeat the last one)
        }
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const uint32_t i = base + lane + u * blockDim.x, nr = i < i1 ? (rec[u].y >> 24) & 127u : 0u;
            uint32_t x[4], m[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) { x[a] = T[rd[u][a]]; m[a] = x[a] % q.B; }
            if (nr <= 4) {
#pragma unroll
                for (int a = 1; a < 4; ++a) {
                    bool value = false, bank = false;
#pragma unroll
                    for (int b = 0; b < a; ++b) { value |= x[b] == x[a]; bank |= m[b] == m[a]; }
                    n += nr > 1 && !value && bank;
                }
            }
            for (uint32_t todo = __ballot_sync(0xffffffffu, nr > 4); todo; todo &= todo - 1) {
                const uint32_t j = base + (__ffs(todo) - 1) + u * blockDim.x;
                const uint32_t u0 = q.op_off[j] + q.ndefs[j], k = q.op_off[j + 1] - u0;
                for (uint32_t a0 = 0; a0 < k; a0 += 32) {
                    const bool mine = a0 + lane < k;
                    const uint32_t ta = mine ? T[q.op_vreg[u0 + a0 + lane]] : 0x10000u + lane, ma = mine ? ta % q.B : ta;
                    bool value = __match_any_sync(0xffffffffu, ta) & below, bank = __match_any_sync(0xffffffffu, ma) & below;
                    for (uint32_t b0 = 0; b0 < a0; b0 += 32) {
                        const uint32_t tb = T[q.op_vreg[u0 + b0 + lane]], mb = tb % q.B;
#pragma unroll 8
                        for (uint32_t b = 0; b < 32; ++b) {
                            value |= __shfl_sync(0xffffffffu, tb, b) == ta;
                            bank |= __shfl_sync(0xffffffffu, mb, b) == ma;
                        }
                    }
                    n += mine && !value && bank;
                }
            }
        }
    }
    return n;
}

// Sources (up to four reads, vreg ids; repeats of a vreg do not count) that hold the register of an earlier source.
__device__ __forceinline__ uint32_t duplicates(const uint32_t (&rd)[4], const uint16_t *T)
{
    uint32_t t[4], n = 0;
#pragma unroll
    for (int a = 0; a < 4; ++a) t[a] = T[rd[a]];
#pragma unroll
    for (int a = 1; a < 4; ++a) {
        bool again = false, same = false;
#pragma unroll
        for (int c = 0; c < a; ++c) {
            again |= rd[c] == rd[a];
            same |= t[c] == t[a];
        }
        n += !again && same;
    }
    return n;
}
// The same for the read at operand a of an instruction whose reads begin at r0.
__device__ __forceinline__ uint32_t duplicate_of(const FParams &q, const uint16_t *T, uint32_t r0, uint32_t a)
{
    const uint32_t v = q.op_vreg[a], t = T[v];
    bool again = false, same = false;
    for (uint32_t c = r0; c < a; ++c) {
        const uint32_t u = q.op_vreg[c];
        again |= u == v;
        same |= T[u] == t;
    }
    return !again && same;
}

// The numbers of the program blocks that the counts of the through-sets need.
__device__ __forceinline__ void load_blocks(const FParams &q, FMisc *M)
{
    const uint32_t b = threadIdx.x;
    if (b > 32) return;
    M->th_off[b] = q.use_th ? q.th_off[min(b, q.nB)] : 0u;
    if (!q.use_th) return;
    const uint32_t i0 = q.blk_off[min(b, q.nB)];
    M->blk_i[b] = i0;
    if (b < q.nB) {
        M->el_n[b] = q.el_count[b];
        M->el_o[b] = q.op_off[i0];
    }
}

// Sources of instruction i in the through-set of block b that hold the register of an earlier source, where an earlier
// source in the through-set holds it too.
__device__ __noinline__ uint32_t member_duplicates(const FParams &q, const uint16_t *T, uint32_t b, uint32_t i)
{
    uint32_t n = 0;
    const uint32_t *th = q.blk_th + (size_t)b * q.Wv;
    const uint32_t r0 = q.op_off[i] + q.ndefs[i], r1 = q.op_off[i + 1];
    for (uint32_t a = r0 + 1; a < r1; ++a) {
        const uint32_t v = q.op_vreg[a];
        if (!((th[v >> 5] >> (v & 31)) & 1u)) continue;
        bool again = false, same = false;
        for (uint32_t c = r0; c < a; ++c) {
            const uint32_t u = q.op_vreg[c];
            again |= u == v;
            same |= ((th[u >> 5] >> (u & 31)) & 1u) && T[u] == T[v];
        }
        n += !again && same;
    }
    return n;
}

template <int NTHR, int BAR>
__device__ __forceinline__ void bar_all()
{
    if constexpr (BAR == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(NTHR) : "memory");
}

// Step 5: the overlaps in the short chunks marked in coll and, for program blocks whose through-set collided, those of the
// definitions without an event, counted exactly; added to M->pairs and M->mind.  With several parts, this block's share.
// The program blocks are taken q.cb at a time (all at once, as a rule: going block by block, the chain of L2 round trips
// in front of the first count took 2 us for each).  cv: [cb][R] words; list: room for nS spans
// (and, LISTED, behind them for the ranges of nC chunks).
// LISTED (k_exact): the bank tally of the table kernel (sources minus banks touched, per instruction) counts a register
// that two source vregs share twice; M->dups receives the number of such sources.  Two sources of an instruction are live
// together in front of it: if they hold the same register, its chunk has collided, or they are both in a through-set that
// has.  And T, W hold nothing yet: what the share needs is fetched here (a hundredth of the vregs, for a row with one
// misplaced vreg; fetching all 10,000 took 30 us).
// LONG: the program's lists are long (EXACT_LONG entries and more on average).
// BAR: the named barrier of the NTHR threads that count (0: they are the whole block).
template <int NTHR, bool LISTED, bool LONG = false, int BAR = 0>
__device__ __forceinline__ void exact_counts(const FParams &q, uint16_t *T, uint8_t *W, uint32_t *cv, const uint32_t *coll,
                                             uint2 *list, FMisc *M, uint32_t part, uint32_t parts, const uint16_t *row)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    uint32_t pairs = 0, mind = 0xFFFFFFFFu, dups = 0;
    for (uint32_t b0 = 0; b0 < q.nB; b0 += q.cb) {
        const uint32_t b1 = min(b0 + q.cb, q.nB);
        const uint32_t s_lo = b0 ? q.blk_short_off[b0] : 0u, s_hi = b1 < q.nB ? q.blk_short_off[b1] : q.nS;
        const uint32_t thcol = q.use_th ? M->thcol : 0u;
        if (tid == 0) M->n_list = M->n_chunks = 0;
        // The through-sets, counted into arrays over the registers: cv[r] = members whose range holds r, plus 65536 for
        // each member whose range starts at r; a range [s, s+w) overlaps (members that hold s) + (members that start at
        // s+1 .. s+w-1).  Members that reach beyond the arrays lie beyond the file: they are compared one by one, with
        // definitions that lie there too.
        if (q.use_th)
            for (uint32_t r = tid; r < (b1 - b0) * q.R; r += NTHR) cv[r] = 0;
        uint4 *chunks = reinterpret_cast<uint4 *>(list + ((q.nS + 1) & ~1u));
        bar_all<NTHR, BAR>();
        for (uint32_t s = s_lo + tid; s < s_hi; s += NTHR)
            if ((coll[s >> 5] >> (s & 31)) & 1u) {
                uint32_t c = 0, c_s0 = 0, c_s1 = 0;
                if (LISTED) {  // a part takes whole chunks
                    c = q.ex.short_chunk[s];
                    if (c % parts != part) continue;
                    c_s0 = q.ex.chunk_short_off[c];
                    c_s1 = q.ex.chunk_short_off[c + 1];
                }
                const uint32_t i0 = q.short_i0[s], b = q.use_th ? q.short_blk[s] - b0 : 0u;
                list[atomicAdd(&M->n_list, 1u)] = make_uint2(i0, (q.short_i0[s + 1] - i0) | (b << 20));
                if (LISTED && s == c_s0) {  // what is occupied when the chunk begins, its operands
                    const uint32_t e0 = q.sen_off[s], o0 = q.op_off[i0];
                    chunks[atomicAdd(&M->n_chunks, 1u)] = make_uint4(e0, q.sen_off[s + 1] - e0, o0, q.op_off[q.short_i0[c_s1]] - o0);
                }
            }
        auto count_member = [&](uint32_t j, uint32_t reg, uint32_t w) {
            uint32_t b = b0;
            while (b + 1 < b1 && M->th_off[b + 1] <= j) ++b;
            if (reg + w <= q.R) {
                uint32_t *c = cv + (b - b0) * q.R + reg;
                atomicAdd(c, 0x10001u);
                for (uint32_t r = 1; r < w; ++r) atomicAdd(c + r, 1u);
            }
        };
        const uint32_t th0 = q.use_th ? M->th_off[b0] : 0u, th1 = q.use_th ? M->th_off[b1] : 0u;
        if (LISTED) {
            // T and W of the n vregs that of(0 .. n - 1) names, by threads first, first + step, ...; then(j, register, width)
            constexpr int FU = 6;
            auto fetch = [&](uint32_t n, uint32_t first, uint32_t step, auto of, auto then) {
                for (uint32_t j0 = first; j0 < n; j0 += FU * step) {
                    uint32_t v[FU], pos[FU], w[FU], t[FU];
#pragma unroll
                    for (int u = 0; u < FU; ++u) v[u] = of(min(j0 + u * step, n - 1));
#pragma unroll
                    for (int u = 0; u < FU; ++u) { pos[u] = q.first_occ[v[u]]; w[u] = q.vinfo[v[u]] & 0xFFu; }
#pragma unroll
                    for (int u = 0; u < FU; ++u) t[u] = row[pos[u] != 0xFFFFFFFFu ? pos[u] : 0u];
#pragma unroll
                    for (int u = 0; u < FU; ++u) {  // (several threads may store the same value)
                        if (pos[u] == 0xFFFFFFFFu) t[u] = 0;
                        T[v[u]] = (uint16_t)t[u];
                        W[v[u]] = (uint8_t)w[u];
                        if (j0 + u * step < n) then(j0 + u * step, t[u], w[u]);
                    }
                }
            };
            auto nothing = [](uint32_t, uint32_t, uint32_t) {};
            fetch(th1 - th0, tid, NTHR, [&](uint32_t j) { return q.th[th0 + j] & 0xFFFFu; },
                  [&](uint32_t j, uint32_t t, uint32_t w) { count_member(th0 + j, t, w); });
            if (tid == 0) { T[q.V] = 0; W[q.V] = 0; }
            bar_all<NTHR, BAR>();
            const uint32_t n_chunks = M->n_chunks;
            if (n_chunks * 512 >= q.V) {
                fetch(q.V, tid, NTHR, [](uint32_t j) { return j; }, nothing);
            } else {  // everything live inside a chunk is occupied when it begins or an operand of it
                for (uint32_t l = tid / (NTHR / 2); l < n_chunks; l += 2) {
                    const uint4 x = chunks[l];
                    fetch(x.y + x.w, tid % (NTHR / 2), NTHR / 2,
                          [&](uint32_t j) { return j < x.y ? q.sen[x.x + j] & 0xFFFFu : q.op_vreg[x.z + j - x.y]; }, nothing);
                }
            }
        } else {
            for (uint32_t j = th0 + tid; j < th1; j += NTHR) {
                const uint32_t v = q.th[j] & 0xFFFFu;
                count_member(j, T[v], W[v]);
            }
        }
        bar_all<NTHR, BAR>();
        const uint32_t n_list = M->n_list;
        // through-set members of block b other than v (itself a member: `member`) that overlap v's range
        auto through_overlaps = [&](uint32_t b, uint32_t v, bool member) {
            const uint32_t s = T[v], w = W[v];
            uint32_t n = 0;
            if (!q.use_th) return n;
            const uint32_t *c = cv + (b - b0) * q.R;
            if (s < q.R) {
                n = (c[s] & 0xFFFFu) - (member && s + w <= q.R ? 1u : 0u);
                for (uint32_t r = s + 1; r < min(s + w, q.R); ++r) n += c[r] >> 16;
            }
            if (s + w > q.P)
                for (uint32_t j = M->th_off[b]; j < M->th_off[b + 1]; ++j) {
                    const uint32_t u = q.th[j] & 0xFFFFu;
                    if (u != v && T[u] + W[u] > q.R && overlap(s, w, T[u], W[u])) ++n;
                }
            return n;
        };
        // A thread takes an instruction: the entries of its live-after list that are not in the through-set, the
        // through-set from the arrays.  The record of the instruction after the next and the first list entries
        // of the next are fetched meanwhile.  (Bound by instruction issue: the lists of loop bodies hold 4 to 10
        // entries, and few of them sit near enough to be looked at more closely.)
        // List entries come four at a time (one request for each entry and lane kept the L1 tags busy for longer than
        // the comparisons take): LQ pieces of the next instruction's list in flight, then LT at a time.
        constexpr int LQ = 3, LT = 4;
        const uint32_t step_unit = NTHR / q.short_len, step_at = NTHR % q.short_len;
        uint32_t unit = tid / q.short_len, at = tid % q.short_len;  // (advances by NTHR instructions)
        auto next_instr = [&](uint32_t &b) -> uint32_t {  // 0xFFFFFFFF: beyond the short chunk, or beyond the list
            uint32_t i = 0xFFFFFFFFu;
            if (unit < n_list) {
                const uint2 span = list[unit];
                if (at < (span.y & 0xFFFFFu)) i = span.x + at;
                b = b0 + (span.y >> 20);
            }
            unit += step_unit;
            at += step_at;
            if (at >= q.short_len) { at -= q.short_len; ++unit; }
            return i;
        };
        auto fetch_rec = [&](uint32_t i) { return q.irec[min(i, q.nI - 1)]; };  // (looked at only if i is one)
        uint32_t rd_nx[4];
        uint4 us_nx[LQ];
        const uint4 *ls4 = reinterpret_cast<const uint4 *>(q.ls);
        auto fetch_list = [&](const uint4 &r) {
            const uint32_t n = r.y & 0xFFFFu, p0 = r.x >> 2, p1 = n ? (r.x + n - 1) >> 2 : p0;
            if (LISTED) {
                const uint32_t nr = (r.y >> 24) & 127u, o = r.w + ((r.y >> 16) & 0xFFu);
#pragma unroll
                for (int u = 0; u < 4; ++u) rd_nx[u] = q.op_vreg[nr ? o + min((uint32_t)u, nr - 1) : 0u];
            }
#pragma unroll
            for (int u = 0; u < LQ; ++u) us_nx[u] = ls4[min(p0 + u, p1)];
        };
        const uint32_t n_slots = n_list * q.short_len;
        if constexpr (LONG) {
            // A warp takes an instruction, its lanes the entries.  (A thread per instruction reads 32 lists at a time, 16 bytes
            // of each.)
            constexpr uint32_t NW = NTHR / 32, LU = 4;
            const uint4 *ls4 = reinterpret_cast<const uint4 *>(q.ls);
            uint32_t unit = (tid >> 5) / q.short_len, at = (tid >> 5) % q.short_len;
            auto next = [&](uint32_t &b) -> uint32_t {
                uint32_t i = 0xFFFFFFFFu;
                if (unit < n_list) {
                    const uint2 span = list[unit];
                    if (at < (span.y & 0xFFFFFu)) i = span.x + at;
                    b = b0 + (span.y >> 20);
                }
                at += NW;
                while (at >= q.short_len) { at -= q.short_len; ++unit; }
                return i;
            };
            uint32_t b_nx = b0, i_nx = next(b_nx);
            uint4 rec_nx = q.irec[min(i_nx, q.nI - 1)];
            for (uint32_t f = tid >> 5; f < n_slots; f += NW) {
                const uint32_t i = i_nx, b = b_nx;
                const uint4 rec = rec_nx;
                i_nx = next(b_nx);
                rec_nx = q.irec[min(i_nx, q.nI - 1)];
                if (i == 0xFFFFFFFFu) continue;
                const uint32_t n = rec.y & 0xFFFFu, nd = (rec.y >> 16) & 0xFFu, p0 = rec.x >> 2, p1 = n ? (rec.x + n - 1) >> 2 : p0;
                uint32_t n_dup = 0;
                for (uint32_t a = rec.w + nd + lane; q.bank_fast && a < q.op_off[i + 1]; a += 32) n_dup += duplicate_of(q, T, rec.w + nd, a);
                n_dup = __reduce_add_sync(0xffffffffu, n_dup);
                if (lane == 0 && n_dup) dups += n_dup - ((thcol >> b) & 1u ? member_duplicates(q, T, b, i) : 0u);
                for (uint32_t d = 0; d < nd; ++d) {
                    const uint32_t v = d ? q.op_vreg[rec.w + d] : rec.z, sv = T[v], wv = W[v];
                    const uint32_t shift = q.wmax - 1 - sv, span = wv + q.wmax - 1;  // (as below)
                    uint32_t cnt = lane ? 0u : through_overlaps(b, v, d ? (q.blk_th[(size_t)b * q.Wv + (v >> 5)] >> (v & 31)) & 1u : rec.y >> 31);
                    for (uint32_t p = p0 + lane; n && p <= p1; p += 32 * LU) {
                        uint4 x4[LU];
#pragma unroll
                        for (uint32_t u = 0; u < LU; ++u) x4[u] = ls4[min(p + u * 32, p1)];
                        uint32_t x[4 * LU], t[4 * LU];
#pragma unroll
                        for (uint32_t u = 0; u < LU; ++u) { x[4 * u] = x4[u].x; x[4 * u + 1] = x4[u].y; x[4 * u + 2] = x4[u].z; x[4 * u + 3] = x4[u].w; }
                        bool near = false;
#pragma unroll
                        for (uint32_t u = 0; u < 4 * LU; ++u) {
                            const bool entry = (p + (u >> 2) * 32) * 4 + (u & 3) - rec.x < n;
                            t[u] = T[entry ? x[u] : q.V];
                            if (!entry) t[u] = 0x1000000u;  // (near nothing)
                            near |= t[u] + shift < span;
                        }
                        if (near) {
#pragma unroll
                            for (uint32_t u = 0; u < 4 * LU; ++u)
                                if (t[u] + shift < span && x[u] != v && t[u] + W[x[u]] > sv) ++cnt;
                        }
                    }
                    for (uint32_t d2 = lane; nd > 1 && d2 < nd; d2 += 32) {  // co-defined vregs that are not live afterwards
                        if (d2 == d || !(q.opflags[rec.w + d2] & OPF_DEAD)) continue;
                        const uint32_t x = q.op_vreg[rec.w + d2];
                        if (overlap(sv, wv, T[x], W[x])) ++cnt;
                    }
                    if (cnt) { pairs += cnt; mind = min(mind, i); }
                }
            }
        } else if (n_slots) {
            uint32_t b_nx = b0, b_nx2 = b0, i_nx = next_instr(b_nx), i_nx2 = next_instr(b_nx2);
            uint4 rec_nx = fetch_rec(i_nx), rec_nx2 = fetch_rec(i_nx2);
            fetch_list(rec_nx);
            for (uint32_t f = tid; f < n_slots; f += NTHR) {
                const uint32_t i = i_nx, b = b_nx;
                const uint4 rec = rec_nx;
                uint32_t us[4 * LQ], ts[4 * LQ], rd[4];
#pragma unroll
                for (int u = 0; u < LQ; ++u) { us[4 * u] = us_nx[u].x; us[4 * u + 1] = us_nx[u].y; us[4 * u + 2] = us_nx[u].z; us[4 * u + 3] = us_nx[u].w; }
#pragma unroll
                for (int u = 0; u < 4; ++u) rd[u] = LISTED ? rd_nx[u] : 0u;
                i_nx = i_nx2;
                b_nx = b_nx2;
                rec_nx = rec_nx2;
                fetch_list(rec_nx);
                i_nx2 = next_instr(b_nx2);
                rec_nx2 = fetch_rec(i_nx2);
                const uint32_t n = rec.y & 0xFFFFu, nd = i != 0xFFFFFFFFu ? (rec.y >> 16) & 0xFFu : 0u;
                if (LISTED && i != 0xFFFFFFFFu && q.bank_fast) {  // (else the tally is made anew)
                    const uint32_t nr = (rec.y >> 24) & 127u;
                    uint32_t n_dup = 0;
                    if (nr <= 4) {  // (missing reads repeat the last one)
                        if (nr > 1) n_dup = duplicates(rd, T);
                    } else {
                        for (uint32_t a = rec.w + nd; a < q.op_off[i + 1]; ++a) n_dup += duplicate_of(q, T, rec.w + nd, a);
                    }
                    // (those of two through-set members are counted with the block's through-set, below)
                    if (n_dup && ((thcol >> b) & 1u)) n_dup -= member_duplicates(q, T, b, i);
                    dups += n_dup;
                }
                if (!nd) continue;
                uint32_t cnt = 0;
                const uint32_t skip = rec.x & 3u;  // (the list begins inside its first piece)
#pragma unroll
                for (int u = 0; u < 4 * LQ; ++u) {
                    const bool entry = (uint32_t)u - skip < n;
                    ts[u] = T[entry ? us[u] : q.V];
                    if (!entry) ts[u] = 0x1000000u;  // (near nothing)
                }
                for (uint32_t d = 0; d < nd; ++d) {
                    const uint32_t v = d ? q.op_vreg[rec.w + d] : rec.z, sv = T[v], wv = W[v];
                    // [t, t + wt) overlaps [sv, sv + wv): t < sv + wv and t > sv - wt, wt at most wmax
                    const uint32_t shift = q.wmax - 1 - sv, span = wv + q.wmax - 1;
                    cnt += through_overlaps(b, v, d ? (q.blk_th[(size_t)b * q.Wv + (v >> 5)] >> (v & 31)) & 1u : rec.y >> 31);
                    bool near = false;
#pragma unroll
                    for (int u = 0; u < 4 * LQ; ++u) near |= ts[u] + shift < span;
                    if (near) {
#pragma unroll
                        for (int u = 0; u < 4 * LQ; ++u)
                            if (ts[u] + shift < span && us[u] != v && ts[u] + W[us[u]] > sv) ++cnt;
                    }
                    for (uint32_t p = (rec.x >> 2) + LQ; p * 4 < rec.x + n; p += LT) {
                        uint4 x4[LT];
#pragma unroll
                        for (int u = 0; u < LT; ++u) x4[u] = ls4[min(p + u, (rec.x + n - 1) >> 2)];
                        uint32_t x[4 * LT], t[4 * LT];
#pragma unroll
                        for (int u = 0; u < LT; ++u) { x[4 * u] = x4[u].x; x[4 * u + 1] = x4[u].y; x[4 * u + 2] = x4[u].z; x[4 * u + 3] = x4[u].w; }
                        bool hit = false;
#pragma unroll
                        for (int u = 0; u < 4 * LT; ++u) {
                            const bool entry = p * 4 + u < rec.x + n;
                            t[u] = T[entry ? x[u] : q.V];
                            if (!entry) t[u] = 0x1000000u;
                        }
#pragma unroll
                        for (int u = 0; u < 4 * LT; ++u) hit |= t[u] + shift < span;
                        if (hit) {
#pragma unroll
                            for (int u = 0; u < 4 * LT; ++u)
                                if (t[u] + shift < span && x[u] != v && t[u] + W[x[u]] > sv) ++cnt;
                        }
                    }
                    if (nd > 1)  // co-defined vregs that are not live after the instruction
                        for (uint32_t d2 = 0; d2 < nd; ++d2) {
                            if (d2 == d || !(q.opflags[rec.w + d2] & OPF_DEAD)) continue;
                            const uint32_t x = q.op_vreg[rec.w + d2];
                            if (overlap(sv, wv, T[x], W[x])) ++cnt;
                        }
                }
                if (cnt) { pairs += cnt; mind = min(mind, i); }
            }
        }
        // In a chunk whose own walk was clean everything that is live is disjoint from the through-set; a
        // definition without an event (a member redefined from itself) overlaps the members that overlap it.
        uint32_t unit_no = 0;  // 4 NTHR entries or instructions; a part takes every parts-th
        for (uint32_t b = b0; b < b1 && thcol; ++b) {
            if (!((thcol >> b) & 1u)) continue;
            const uint32_t n_el = M->el_n[b];
            const uint4 *el = q.el + M->el_o[b];  // instruction, chunk, vreg | member << 31, short chunk
            for (uint32_t u0 = 0; u0 < n_el; u0 += 4 * NTHR) {
                if (unit_no++ % parts != part) continue;
                const uint32_t e0 = u0 + tid;
                uint4 x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = el[min(e0 + u * NTHR, n_el - 1)];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (e0 + u * NTHR >= n_el || !(x[u].z >> 31) || ((coll[x[u].w >> 5] >> (x[u].w & 31)) & 1u)) continue;
                    const uint32_t n = through_overlaps(b, x[u].z & 0xFFFFu, true);
                    if (n) { pairs += n; mind = min(mind, x[u].x); }
                }
            }
            if (!LISTED) continue;
            // sources of the block's instructions that are both in the through-set
            const uint32_t i1 = M->blk_i[b + 1];
            for (uint32_t u0 = M->blk_i[b]; u0 < i1; u0 += 4 * NTHR) {
                if (unit_no++ % parts != part) continue;
                const uint32_t i0 = u0 + tid;
                uint4 rec[4];
                uint32_t rd[4][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) rec[u] = q.irec[min(i0 + u * NTHR, i1 - 1)];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t nr = (rec[u].y >> 24) & 127u, o = rec[u].w + ((rec[u].y >> 16) & 0xFFu);
#pragma unroll
                    for (int r = 0; r < 4; ++r) rd[u][r] = q.op_vreg[nr ? o + min((uint32_t)r, nr - 1) : 0u];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t i = i0 + u * NTHR, nr = (rec[u].y >> 24) & 127u;
                    if (i >= i1 || nr < 2) continue;
                    if (nr > 4 || duplicates(rd[u], T)) dups += member_duplicates(q, T, b, i);
                }
            }
        }
        bar_all<NTHR, BAR>();
    }
    pairs = __reduce_add_sync(0xffffffffu, pairs);
    mind = __reduce_min_sync(0xffffffffu, mind);
    if (LISTED) {
        dups = __reduce_add_sync(0xffffffffu, dups);
        if (lane == 0 && dups) atomicAdd(&M->dups, dups);
    }
    if (lane == 0 && pairs) {
        atomicAdd(&M->pairs, pairs);
        atomicMin(&M->mind, mind);
    }
    bar_all<NTHR, BAR>();
}

// What the kernels read of a program.
inline FParams fused_params(const vl_program *p, bool dict)
{
    FParams q{};
    q.nI = p->nI; q.V = p->V; q.nO = dict ? p->nD : p->nO; q.P = p->P; q.B = p->B; q.nB = p->nB; q.nS = p->nS; q.Wv = p->Wv;
    q.Wp = (p->P + p->wmax + 31) / 32; q.R = p->P + p->wmax + 2; q.wmax = p->wmax;
    q.bank_fast = p->bank_fast; q.use_th = p->use_th;
    q.short_len = p->short_len;
    q.first_occ = dict ? p->d_dict_first_occ : p->d_first_occ; q.vreg16 = dict ? p->d_dict_vreg16 : p->d_vreg16;
    q.vinfo = p->d_vinfo; q.first_def_instr = p->d_first_def_instr; q.op_off = p->d_op_off; q.op_vreg = p->d_op_vreg;
    q.entry_instr = dict ? p->d_dict_instr : nullptr; q.ndefs = p->d_ndefs; q.opflags = p->d_opflags;
    q.vcons = p->d_vcons; q.rs_prefix = p->d_rs_prefix; q.bank_list = p->d_bank_list;
    for (int c = 0; c < 4; ++c) q.bank_seg[c] = p->bank_seg[c];
    q.th_off = p->d_th_off; q.th = p->d_th; q.blk_th = p->d_blk_th; q.sev_off = p->d_sev_off; q.sev = p->d_sev;
    q.sen_off = p->d_sen_off; q.sen = p->d_sen;
    q.short_blk = p->d_short_blk; q.short_i0 = p->d_short_i0; q.blk_short_off = p->d_blk_short_off;
    q.ls = p->d_ls; q.irec = p->d_irec; q.blk_off = p->d_blk_off;
    q.el = p->d_el; q.el_count = p->d_el_count;
    return q;
}

}  // namespace
