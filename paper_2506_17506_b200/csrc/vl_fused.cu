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

#include "vl_internal.cuh"

#define EXACT_NT 256
#define EXACT_SMEM (224u * 1024)  // shared memory of a block of k_exact, at most
#define EXACT_ROWS 2000           // rows that k_fused leaves counts of, at most: their items fit 16 bits

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

// The jobs of up to N programs in one grid: blockIdx.y is the program.
template <int N>
struct FMany {
    FParams p[N];
};
static_assert(sizeof(FMany<VL_FUSED_MANY>) <= 32764, "kernel arguments");

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
template <int NTHR, bool LISTED, bool LONG = false>
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
        __syncthreads();
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
            __syncthreads();
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
        __syncthreads();
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
        __syncthreads();
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
    __syncthreads();
}

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
                cs[CS_ITEMS] = exact_parts(chunks, EXACT_PART_CHUNKS) | exact_parts(chunks, EXACT_FINE_CHUNKS) << 16;
            }
        } else if (lane == 0) {
            if (HAND) q.ex.cstate[k * 8 + CS_ITEMS] = 0;
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
// ROWS: the candidates are the rows of k_fused, which left the number of items of each in cstate; every block adds them up
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
        __shared__ uint32_t s_sum[EXACT_NT / 32];
        const uint32_t per = (q.ex.rows + EXACT_NT - 1) / EXACT_NT, k0 = tid * per, k1 = min(k0 + per, q.ex.rows);
        uint32_t n = 0;  // of this thread's rows, coarse | fine << 16 (at most EXACT_ROWS rows: neither half overflows)
        for (uint32_t k = k0; k < k1; ++k) {
            const uint32_t x = q.ex.cstate[(size_t)k * 8 + CS_ITEMS];
            first[k] = x;
            n += x;
        }
        uint32_t inc = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= (uint32_t)d) inc += y;
        }
        if (lane == 31) s_sum[tid >> 5] = inc;
        __syncthreads();
        uint32_t before = inc - n, all = 0;
#pragma unroll
        for (uint32_t w = 0; w < EXACT_NT / 32; ++w) {
            if (w < tid >> 5) before += s_sum[w];
            all += s_sum[w];
        }
        const uint32_t shift = all >> 16 <= q.ex.fine_items ? 16u : 0u;
        n_items = (all >> shift) & 0xFFFFu;
        uint32_t at = (before >> shift) & 0xFFFFu;
        for (uint32_t k = k0; k < k1; ++k) {
            const uint32_t x = (first[k] >> shift) & 0xFFFFu;
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
            if (tid == 0) M->bank = (part == 0 ? cs[CS_BANK] : 0u) - (ROWS ? 0u : M->dups);
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

// What the kernels of this file read of a program.
FParams fused_params(const vl_program *p, bool dict)
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

bool vl_fused_wanted(vl_program *p, uint64_t K)
{
    if (p->group_opt || p->threads_opt || p->test_wait) return false;  // the caller asks for the batched kernels
    if (!vl_verify_takes(p)) return false;                             // (refused, however few the rows)
    if (p->known[VL_KNOWN_SEN] >= FUSED_MANY_ENTRIES && (K < FUSED_FEW_ROWS || K > (uint64_t)vl_sm_count(p) || long_lists(p))) return false;
    const FPlan pl = fused_plan(p, K);
    if (!pl.threads) return false;
    const uint64_t resident = (uint64_t)pl.bpm * vl_sm_count(p);
    const uint64_t rounds = (K + resident - 1) / resident;
    return rounds <= 1 || rounds * (6000 + 7ull * p->nI) <= 72000;
}

// Programs of at least that many instructions whose rows share multiprocessors hand the exact counts to k_exact: a row that
// fails used to keep its few warps busy for longer than all the rest took, now every multiprocessor shares in it.  300 rows
// of 8,000 instructions 45 us against 88 with 10 % of the rows failing, of 11,317 instructions 62 against 90; with none
// failing the second launch costs 1 us (32.9, 46.0).  Of 5,000 instructions it gains nothing (46.4 against 43.1, 48.2 against
// 48.5 with 30 % failing), nor do rows that have a multiprocessor to themselves (50 rows of 11,317 instructions 22 us).
#define FUSED_HAND_INSTRS 7000u

// What k_fused and k_exact share.
static int hand_scratch(vl_program *p, int slot, uint64_t rows, VlExactArgs *ex)
{
    ex->rows = (uint32_t)rows;
    vl_program::VScratch &v = p->fs[slot];
    const uint64_t aw = (p->nC + 31) / 32;
    if (v.rows < rows || v.aw != aw) {
        VL_CUDA(p, cudaFree(v.block));
        v = vl_program::VScratch{};
        rows = std::max<uint64_t>(rows, 3ull * vl_sm_count(p));
        VL_CUDA(p, cudaMalloc(&v.block, rows * (8 + 4 + aw) * 4));
        v.cstate = static_cast<uint32_t *>(v.block); v.racc = v.cstate + rows * 8; v.anom = v.racc + rows * 4;
        v.rows = rows; v.aw = aw;
    }
    ex->cstate = v.cstate; ex->racc = v.racc; ex->anom = v.anom;
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
            const int rc = hand_scratch(p0, slot, rows, &ex);
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
    return vl_fused_wanted(p, K) && fused_smem(p, 256).total <= 48 * 1024;
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
