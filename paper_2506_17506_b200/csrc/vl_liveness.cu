// Liveness on the GPU and the per-program tables the verify kernels consume.
//
// Every block is cut into chunks (the unit of the verify walk), every chunk into pieces of at most
// PIECE_INSTRS instructions (the unit of the instruction-level work here), and runs of pieces of one chunk
// form short chunks (the unit of the one-candidate walk).  A run of a longer program is five launches:
//   k_sets     read/write bitsets of every piece, composed to its chunk's (one thread block per chunk)
//   k_flow     per 32 words of the bitsets: block sets, fixed point over the blocks, live sets at the
//              chunk boundaries (bitset words are independent of each other)
//   k_count    live sets at the piece boundaries; live-after list lengths, operand flags, walk-event
//              counts and the vregs whose occupancy changes (one thread block per chunk)
//   k_offsets  through-sets, entry counts; the last thread block makes every offset and leaves the totals
//              and the status word in pinned host memory
//   k_fill     live-after lists in CSR form, walk events, through-set lists, side by side in one grid
// and of a program of up to LIVE_SMALL_INSTRS instructions two: k_small (the first four by one cluster) and k_fill.
// What bounds a run is the chain of launches and of L2 round trips inside them, not the bytes (34 MB of
// lists for 32,000 instructions): the lanes of a warp take the operands of a piece, and a kernel's blocks start while the
// kernel before it drains.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include <cooperative_groups.h>

#include "vl_internal.cuh"

#define NT 128  // threads per block of the operand-table kernels
#define PIECE_INSTRS 8         // instructions of a piece, at most
#define PC_WARPS 20            // warps per block of k_sets and k_count: the pieces of a chunk of the default size at once
#define PC_NT (PC_WARPS * 32)
#define PIECE_OPERANDS 32      // and its operands, one per lane, unless its instructions have many (vl_layout)
#define LV_WARPS 8             // warps per block of k_fill
#define LV_NT (LV_WARPS * 32)
#define FILL_WARP_WORDS (32 + 1024 + 256)  // shared memory of a warp of k_fill behind its two bitsets
#define FLOW_WARPS 16          // warps per block of k_flow
#define OFF_NT 256             // threads per block of k_offsets
#define SEG_CHUNKS 8           // chunks that a warp of k_flow composes in one go (longer in very long programs)
#define SHORT_CHUNKS 512       // short chunks per program aimed at: the threads of one block of the one-candidate walk

#define SMALL_NT 512
#define SMALL_WARPS (SMALL_NT / 32)
#define SMALL_BLOCKS 8         // thread blocks of a cluster (the portable size)
#define SMALL_ONE_PIECES 32    // pieces up to which one thread block takes the program
#define SMALL_SMEM (160 * 1024)   // shared memory of a thread block, at most
#define LIVE_SMALL_INSTRS 4096    // instructions of a program, at most

// Where the parts of a block's shared memory begin in k_small, in words, and how much there is.  (Made on the host: the kernel
// reads them as constants; computed there, from seven numbers, they cost more instructions than the work between them.)
struct SmallSmem {
    uint16_t clo, pi, po, pc, xs, fl, pu, pd, cu, cd, bu, bd, bi, bo, bt, lo, ev, plo, pev, cev, cent, sent, sev, thn, rd;
    uint16_t tab, tab_words, blk_chunk, chunk_piece, chunk_blk, chunk_short, short_piece, short_chunk, blk_off, succ_off, succ;  // layout tables
    // bytes; pieces, ops: of the largest share
    uint32_t init(uint32_t nB, uint32_t nE, uint32_t nC, uint32_t nS, uint32_t Wv, uint32_t pieces, uint32_t ops)
    {
        uint64_t at = 0;
        auto take = [&](uint64_t n) { const uint64_t x = at; at += (n + 1) & ~1ull; return (uint16_t)x; };
        clo = take(2 * nC);                                          // list entries per chunk (64 bit)
        tab = take(0);
        // (side by side, as vl_layout has them)
        auto table = [&](uint64_t n) { const uint64_t x = at; at += (n + 4) & ~3ull; return (uint16_t)x; };
        blk_chunk = table(nB + 1); chunk_piece = table(nC + 1); chunk_blk = table(nC); chunk_short = table(nC + 1); short_piece = table(nS);
        short_chunk = table(nS); blk_off = table(nB + 1); succ_off = table(nB + 1); succ = table(nE);
        tab_words = (uint16_t)(at - tab);
        pi = take(pieces + 1); po = take(pieces + 1); pc = take(pieces);  // first instructions and operands of the share's pieces, their chunks
        xs = take(ops); fl = take((ops + 3) / 4);                    // operands and their flags (a byte each)
        const uint64_t PW = (uint64_t)pieces * Wv, CW = (uint64_t)nC * Wv, BW = (uint64_t)nB * Wv;
        pu = take(PW); pd = take(PW);                                // sets of the share's pieces; pu: then live after the piece
        cu = take(CW); cd = take(CW);                                // sets of every chunk; cu: then live before the chunk
        bu = take(BW); bd = take(BW); bi = take(BW); bo = take(BW); bt = take(BW);  // of every block; bt: touched
        lo = take(pieces * PIECE_INSTRS); ev = take(pieces * PIECE_INSTRS);  // per instruction: entries and events before it in its piece
        plo = take(pieces); pev = take(pieces);                      // of the pieces; then before them in their chunk
        cev = take(nC); cent = take(nC); sent = take(nS); sev = take(nS); thn = take(nB);
        rd = take((uint64_t)SMALL_WARPS * Wv);                       // a set per warp, for pieces of more than 32 operands
        return at > SMALL_SMEM / 4 ? 0xFFFFFFFFu : (uint32_t)at * 4;
    }
};

// Everything the kernels of a run read and write.
struct LiveArgs {
    uint32_t nB, nI, V, nE, Wv, nC, nP, nS, nSeg;
    int use_th, wide_smem;
    // program and layout
    const uint32_t *op_off, *op_vreg, *succ_off, *succ, *blk_off;
    const uint8_t *ndefs, *width;
    const uint32_t *chunk_i0, *chunk_i1, *chunk_blk, *blk_chunk_off, *piece_i0, *piece_o0, *op_word, *piece_chunk, *chunk_piece_off;
    const uint32_t *seg_c0, *blk_seg_off;         // segments of k_flow: runs of chunks of one block
    const uint32_t *short_p0, *chunk_short_off;   // short chunks: first piece of each; short chunks of every chunk
    // working sets
    uint32_t *piece_use, *piece_def, *piece_end, *chunk_use, *chunk_def, *chunk_end, *chunk_entry, *blk_touch;
    uint32_t *lo_rel, *ev_rel;                    // per instruction: list entries / events before it in its chunk
    unsigned long long *chunk_lo;                 // per chunk: list entries of its instructions
    uint32_t *chunk_ev, *chunk_lo0;               // events of its instructions; first list entry
    uint32_t *centry_cnt, *short_ent, *short_ev;  // entry events per chunk, per short chunk; other events per short chunk
    uint32_t *flow_scratch;                       // k_flow's working set when it does not fit shared memory
    uint32_t *counters;                           // [0] blocks of k_offsets that have finished
    const uint4 *share;                           // k_small: shares of the thread blocks, tables for shared memory
    const uint32_t *small_tab;
    SmallSmem small;
    // results
    uint32_t *blk_in, *blk_out, *lo_off, *lo, *ls, *ls_adj, *blk_th, *th_cnt, *th_off, *th, *cev_off, *ev8, *sev_off, *sev, *sen_off, *sen;
    uint8_t *opflags;
    uint4 *ev, *el, *irec;
    uint32_t *el_count, *status;
    uint32_t *host_out;                           // pinned: [0] status, [2..] totals (64 bit)
};
// The runs of up to N programs in one grid: blockIdx.y is the program.  (As kernel arguments: 64 programs of one call
// would otherwise be 320 launches, or an upload in front of every run.)
#define LV_MANY 48
template <int N>
struct LiveMany {
    LiveArgs p[N];
};
static_assert(sizeof(LiveMany<LV_MANY>) <= 32764, "kernel arguments");
#define LIVE_ARGS const LiveArgs &q = a.p[N == 1 ? 0 : blockIdx.y]

enum { LV_TOT_LO = 0, LV_TOT_EV = 1, LV_TOT_TH = 2, LV_TOT_LS = VL_KNOWN_LS, LV_TOT_SEV = 4, LV_TOT_SEN = VL_KNOWN_SEN, LV_TOTALS = 6 };

// ------------------------------------------------------------------ device helpers
__device__ __forceinline__ bool bit_get(const uint32_t *s, uint32_t v) { return (s[v >> 5] >> (v & 31)) & 1u; }

// Exclusive scan over the threads of a block (a whole number of warps, at most 32), any integer type;
// *total gets the block sum.  s_scan needs 34 elements.  Contains barriers.
template <typename T>
__device__ T block_excl_scan(T x, T *s_scan, T *total)
{
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= (uint32_t)d) inc += y;
    }
    __syncthreads();  // protects s_scan against readers of a previous call
    if (lane == 31) s_scan[w] = inc;
    __syncthreads();
    if (w == 0) {
        const T t = lane < nw ? s_scan[lane] : (T)0;
        T ti = t;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const T y = __shfl_up_sync(0xffffffffu, ti, d);
            if (lane >= (uint32_t)d) ti += y;
        }
        if (lane < nw) s_scan[lane] = ti - t;
        if (lane == 31) s_scan[33] = ti;
    }
    __syncthreads();
    *total = s_scan[33];
    return s_scan[w] + inc - x;
}

// An operand of a piece as a word: vreg (16 bits), instruction inside the piece (4 bits at 16), and how it meets the piece's
// other operands, which the layout of the program fixes (k_operand_words; found anew in every run, by shuffles or matches of
// a warp's lanes, it took k_sets and k_count half of their time).  In a piece of more than PIECE_OPERANDS operands only OW_DEF
// and OW_EXPOSED are set.
enum : uint32_t {
    OW_DEF = 1u << 20,      // definition
    OW_DUP = 1u << 21,      // read: an earlier read of the instruction has the vreg
    OW_OTHER = 1u << 22,    // the instruction's other side (reads / writes) has the vreg
    OW_EXPOSED = 1u << 23,  // read: no earlier instruction of the piece writes the vreg
    OW_LATER = 1u << 24,    // a later instruction of the piece touches the vreg ...
    OW_READ = 1u << 25,     // ... and the first such reads it
    OW_MANY = 1u << 26      // the instruction has several definitions
};
struct Piece {
    uint32_t i0, ni, o0, n;  // first instruction, instructions; first operand, operands
    __device__ __forceinline__ void init(const LiveArgs &q, uint32_t p)
    {
        i0 = q.piece_i0[p];
        o0 = q.piece_o0[p];
        ni = q.piece_i0[p + 1] - i0;
        n = q.piece_o0[p + 1] - o0;
    }
    // operand j of the piece, 0 beyond it
    __device__ __forceinline__ uint32_t get(const LiveArgs &q, uint32_t j) const { return j < n ? q.op_word[o0 + j] : 0u; }
};
__device__ __forceinline__ uint32_t po_vreg(uint32_t x) { return x & 0xFFFFu; }
__device__ __forceinline__ uint32_t po_instr(uint32_t x) { return (x >> 16) & 15u; }
__device__ __forceinline__ bool po_def(uint32_t x) { return x & OW_DEF; }
__device__ __forceinline__ uint32_t low_bits(uint32_t n) { return n >= 32 ? 0xFFFFFFFFu : (1u << n) - 1u; }

// Lanes whose operand belongs to the same instruction (every lane of the warp; 4 ballots at 26 cycles each, a match
// instruction takes 380 cycles alone and 1,080 beside 15 other warps).
__device__ __forceinline__ uint32_t same_instr(uint32_t x, bool mine)
{
    uint32_t same = __ballot_sync(0xffffffffu, mine);
#pragma unroll
    for (int j = 16; j < 19; ++j) {
        const uint32_t bit = __ballot_sync(0xffffffffu, (x >> j) & 1u);
        same &= (x >> j) & 1u ? bit : ~bit;
    }
    return same;
}

// ============================================================================ k_sets
// One thread block per chunk.  use = vregs read before any write inside the piece (the chunk), def = vregs written.
// Read and write sets of one piece, into empty bitsets of shared memory (a warp; x: its first 32 operands, one per lane).
__device__ __forceinline__ void piece_sets(const LiveArgs &q, const Piece &po, uint32_t x, uint32_t lane, uint32_t *s_use, uint32_t *s_def)
{
    for (uint32_t j = lane; j < po.n; j += 32) {
        const uint32_t y = j == lane ? x : po.get(q, j);
        if (y & (OW_DEF | OW_EXPOSED)) atomicOr(&(po_def(y) ? s_def : s_use)[po_vreg(y) >> 5], 1u << (y & 31));
    }
}

template <int N>
__global__ void __launch_bounds__(PC_NT) k_sets(const __grid_constant__ LiveMany<N> a)
{
    LIVE_ARGS;
    extern __shared__ uint32_t sm[];
    const uint32_t c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_wait();
    pdl_go();
    // what later kernels of the run update with atomics starts at zero
    for (size_t i = (size_t)c * blockDim.x + tid; i < (size_t)q.nB * q.Wv; i += (size_t)gridDim.x * blockDim.x) q.blk_touch[i] = 0;
    for (uint32_t b = c * blockDim.x + tid; b < q.nB; b += gridDim.x * blockDim.x) q.el_count[b] = 0;
    if (c == 0 && tid == 0) { q.counters[0] = 0; *q.status = 0; }
    if (c >= q.nC) return;
    uint32_t *s_use = sm + (size_t)warp * 2 * q.Wv, *s_def = s_use + q.Wv;
    const uint32_t p0 = q.chunk_piece_off[c], p1 = q.chunk_piece_off[c + 1];
    for (uint32_t p = p0 + warp; p < p1; p += blockDim.x / 32) {
        Piece po;
        po.init(q, p);
        const uint32_t x = po.get(q, lane);
        for (uint32_t w = lane; w < 2 * q.Wv; w += 32) s_use[w] = 0;
        __syncwarp();
        piece_sets(q, po, x, lane, s_use, s_def);
        __syncwarp();
        for (uint32_t w = lane; w < q.Wv; w += 32) {
            q.piece_use[(size_t)p * q.Wv + w] = s_use[w];
            q.piece_def[(size_t)p * q.Wv + w] = s_def[w];
        }
        __syncwarp();
    }
    __syncthreads();
    for (uint32_t w = tid; w < q.Wv; w += blockDim.x) {
        uint32_t u = 0, d = 0;
#pragma unroll 4
        for (uint32_t p = p0; p < p1; ++p) {
            u |= q.piece_use[(size_t)p * q.Wv + w] & ~d;
            d |= q.piece_def[(size_t)p * q.Wv + w];
        }
        q.chunk_use[(size_t)c * q.Wv + w] = u;
        q.chunk_def[(size_t)c * q.Wv + w] = d;
    }
}

// ============================================================================ k_flow
// Backward dataflow to the least fixed point.  A thread block takes 32 words of every bitset (one per lane);
// bitset words are independent of each other, so nothing is exchanged between thread blocks.  Warps compose
// the chunk sets of segments (SEG_CHUNKS loads in flight instead of a chain over a block's chunks), one warp
// iterates the blocks, and the warps walk the segments back to the live sets at the chunk boundaries.
// Working set: [4][nB][32] + [2][nSeg][32] words and the successor lists, in shared memory or flow_scratch.
template <int N>
__global__ void __launch_bounds__(FLOW_WARPS * 32) k_flow(const __grid_constant__ LiveMany<N> a)
{
    LIVE_ARGS;
    extern __shared__ uint32_t sm[];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t w = blockIdx.x * 32 + lane;
    if (blockIdx.x * 32 >= q.Wv) return;
    const bool in = w < q.Wv;
    const size_t words = ((size_t)4 * q.nB + 2 * (size_t)q.nSeg) * 32 + q.nB + 1 + q.nE;
    uint32_t *base = q.flow_scratch ? q.flow_scratch + blockIdx.x * words : sm;
    uint32_t *s_use = base, *s_def = s_use + (size_t)q.nB * 32, *s_in = s_def + (size_t)q.nB * 32,
             *s_out = s_in + (size_t)q.nB * 32, *seg_u = s_out + (size_t)q.nB * 32, *seg_d = seg_u + (size_t)q.nSeg * 32,
             *s_so = seg_d + (size_t)q.nSeg * 32, *s_su = s_so + q.nB + 1;
    for (uint32_t i = tid; i <= q.nB; i += FLOW_WARPS * 32) s_so[i] = q.succ_off[i];
    for (uint32_t i = tid; i < q.nE; i += FLOW_WARPS * 32) s_su[i] = q.succ[i];
    pdl_go();
    pdl_wait();
    for (uint32_t s = warp; s < q.nSeg; s += FLOW_WARPS) {
        const uint32_t c1 = q.seg_c0[s + 1];
        uint32_t u = 0, d = 0;
        for (uint32_t c0 = q.seg_c0[s]; c0 < c1; c0 += SEG_CHUNKS) {
            uint32_t cu[SEG_CHUNKS], cd[SEG_CHUNKS];
#pragma unroll
            for (int j = 0; j < SEG_CHUNKS; ++j) {
                const bool ok = in && c0 + j < c1;
                cu[j] = ok ? q.chunk_use[(size_t)(c0 + j) * q.Wv + w] : 0u;
                cd[j] = ok ? q.chunk_def[(size_t)(c0 + j) * q.Wv + w] : 0u;
            }
#pragma unroll
            for (int j = 0; j < SEG_CHUNKS; ++j) { u |= cu[j] & ~d; d |= cd[j]; }
        }
        seg_u[s * 32 + lane] = u;
        seg_d[s * 32 + lane] = d;
    }
    __syncthreads();
    for (uint32_t b = warp; b < q.nB; b += FLOW_WARPS) {
        uint32_t u = 0, d = 0;
        for (uint32_t s = q.blk_seg_off[b]; s < q.blk_seg_off[b + 1]; ++s) { u |= seg_u[s * 32 + lane] & ~d; d |= seg_d[s * 32 + lane]; }
        s_use[b * 32 + lane] = u;
        s_def[b * 32 + lane] = d;
        s_in[b * 32 + lane] = 0;
        s_out[b * 32 + lane] = 0;
    }
    __syncthreads();
    if (warp == 0) {
        bool changed = true;
        for (uint32_t sweep = 0; sweep < q.nB + 2 && __any_sync(0xffffffffu, changed); ++sweep) {
            changed = false;
            for (uint32_t b = q.nB; b-- > 0;) {
                uint32_t o = 0;
                for (uint32_t e = s_so[b]; e < s_so[b + 1]; ++e) o |= s_in[s_su[e] * 32 + lane];
                const uint32_t i = s_use[b * 32 + lane] | (o & ~s_def[b * 32 + lane]);
                if (o != s_out[b * 32 + lane] || i != s_in[b * 32 + lane]) changed = true;
                s_out[b * 32 + lane] = o;
                s_in[b * 32 + lane] = i;
            }
        }
        uint32_t st = changed ? (uint32_t)ST_NO_CONVERGE : 0u;
        if (s_in[lane] != 0) st |= ST_NOT_STRICT;  // block 0 is the entry
        st = __reduce_or_sync(0xffffffffu, st);
        if (st && lane == 0) atomicOr(q.status, st);
    }
    __syncthreads();
    for (uint32_t b = warp; b < q.nB; b += FLOW_WARPS) {
        uint32_t live = s_out[b * 32 + lane];
        if (in) {
            q.blk_in[(size_t)b * q.Wv + w] = s_in[b * 32 + lane];
            q.blk_out[(size_t)b * q.Wv + w] = live;
        }
        for (uint32_t s = q.blk_seg_off[b + 1]; s-- > q.blk_seg_off[b];) {  // seg_u becomes the live set behind the segment
            const uint32_t u = seg_u[s * 32 + lane], d = seg_d[s * 32 + lane];
            seg_u[s * 32 + lane] = live;
            live = u | (live & ~d);
        }
    }
    __syncthreads();
    for (uint32_t s = warp; s < q.nSeg; s += FLOW_WARPS) {
        uint32_t live = seg_u[s * 32 + lane];
        const uint32_t c_lo = q.seg_c0[s];
        for (uint32_t c1 = q.seg_c0[s + 1]; c1 > c_lo;) {
            uint32_t cu[SEG_CHUNKS], cd[SEG_CHUNKS];
#pragma unroll
            for (int j = 0; j < SEG_CHUNKS; ++j) {
                const bool ok = in && c1 - c_lo > (uint32_t)j;
                cu[j] = ok ? q.chunk_use[(size_t)(c1 - 1 - j) * q.Wv + w] : 0u;
                cd[j] = ok ? q.chunk_def[(size_t)(c1 - 1 - j) * q.Wv + w] : 0u;
            }
#pragma unroll
            for (int j = 0; j < SEG_CHUNKS; ++j)
                if (in && c1 - c_lo > (uint32_t)j) {
                    q.chunk_end[(size_t)(c1 - 1 - j) * q.Wv + w] = live;
                    live = cu[j] | (live & ~cd[j]);
                    q.chunk_entry[(size_t)(c1 - 1 - j) * q.Wv + w] = live;
                }
            c1 -= min(c1 - c_lo, (uint32_t)SEG_CHUNKS);
        }
    }
}

// An operand's flags, and the walk events that it makes.  many: the instruction has several definitions; lv: its vreg is live
// after the instruction; dup: an earlier read of the instruction has the vreg; other: the instruction's other side
// (reads / writes) has it.
__device__ __forceinline__ uint32_t operand_events(bool many, bool def, bool lv, bool dup, bool other, uint32_t *flags)
{
    if (!def) {
        const bool kill = !dup && !lv;  // a read of a vreg that stays live releases nothing
        *flags = (kill ? OPF_KILL : 0) | (dup ? OPF_DUP : 0);
        return kill ? 1u : 0u;
    }
    const bool elide = other && lv, post = !lv && many;
    *flags = OPF_DEF | (elide ? OPF_ELIDE : 0) | ((lv || many) ? OPF_SET : 0) | (post ? OPF_POST : 0) | (lv ? 0 : OPF_DEAD);
    return elide ? 0u : 1u + (post ? 1u : 0u);
}

// The operands of a piece of at most 32, one per lane: flags, touched vregs, and per instruction the events (s_ev) and what it
// adds to the live count going backwards (s_d).  An operand's vreg is live after its instruction iff the next instruction of
// the piece that touches it reads it, or, if none does, iff it is live after the piece (end).  touched: what this lane's word
// of touch is known to hold.
__device__ __forceinline__ void count_narrow(const Piece &po, uint32_t x, const uint32_t *end, uint8_t *opflags, uint32_t *touch,
                                             uint32_t touched, int *s_d, uint32_t *s_ev)
{
    const uint32_t lane = threadIdx.x & 31, v = po_vreg(x);
    const bool mine = lane < po.n, def = po_def(x);
    if (lane < PIECE_INSTRS) { s_d[lane] = 0; s_ev[lane] = 0; }
    bool up = false, down = false;
    uint32_t evs = 0;
    if (mine) {
        const bool lv = x & OW_LATER ? (x & OW_READ) != 0 : (end[v >> 5] >> (v & 31)) & 1u;
        const bool dup = x & OW_DUP, other = x & OW_OTHER;
        uint32_t flags;
        evs = operand_events(x & OW_MANY, def, lv, dup, other, &flags);
        opflags[lane] = (uint8_t)flags;
        // a read: live before the instruction, but not among what is live behind it and not written by it
        up = !def && !dup && !(lv && !other);
        down = def && lv;
        if (evs && !((touched >> (v & 31)) & 1u)) atomicOr(&touch[v >> 5], 1u << (v & 31));
    }
    const uint32_t here = same_instr(x, mine);
    const uint32_t ups = __ballot_sync(0xffffffffu, up), downs = __ballot_sync(0xffffffffu, down);
    const uint32_t ev1 = __ballot_sync(0xffffffffu, evs != 0), ev2 = __ballot_sync(0xffffffffu, evs > 1);
    __syncwarp();
    if (mine && lane == __ffs(here) - 1) {
        s_d[po_instr(x)] = (int)__popc(ups & here) - (int)__popc(downs & here);
        s_ev[po_instr(x)] = __popc(ev1 & here) + __popc(ev2 & here);
    }
}

// The same for a piece with more operands: instruction by instruction, from the last to the first.  reads: an empty bitset of
// this warp's own; live: one for the live set (null: the piece is a single instruction).
// (200 instructions of 60 reads 172 us for the run, all operands met in pairs 976; 100 of 100 definitions 202 and 2,133)
template <bool GLOBAL>  // touch lies in global memory
__device__ __noinline__ void count_wide(const LiveArgs &q, const Piece &po, const uint32_t *end, volatile uint32_t *reads,
                                        volatile uint32_t *live, uint8_t *opflags, uint32_t *touch, int *s_d, uint32_t *s_ev)
{
    const uint32_t lane = threadIdx.x & 31;
    auto has = [](const volatile uint32_t *s, uint32_t v) { return (s[v >> 5] >> (v & 31)) & 1u; };
    if (live) {
        for (uint32_t w = lane; w < q.Wv; w += 32) live[w] = end[w];
        __syncwarp();
    }
    const volatile uint32_t *after = live ? live : end;
    for (uint32_t k = po.ni; k-- > 0;) {
        const uint32_t o0 = q.op_off[po.i0 + k], nd = q.ndefs[po.i0 + k], r0 = o0 + nd, o1 = q.op_off[po.i0 + k + 1];
        uint32_t n_ev = 0;
        auto event = [&](uint32_t v, uint32_t n) {
            const uint32_t bit = 1u << (v & 31);
            n_ev += n;
            if (n && (!GLOBAL || !(__ldcg(&touch[v >> 5]) & bit))) atomicOr(&touch[v >> 5], bit);
        };
        for (uint32_t o = r0; o < o1; o += 32) {  // which reads are the first of their vreg
            const bool mine = o + lane < o1;
            const uint32_t v = mine ? q.op_vreg[o + lane] : 0x10000u + lane;
            const uint32_t same = __match_any_sync(0xffffffffu, v);
            const bool dup = mine && ((same & low_bits(lane)) || has(reads, v));
            __syncwarp();
            if (mine) {
                uint32_t flags;
                if (!dup) atomicOr(const_cast<uint32_t *>(reads) + (v >> 5), 1u << (v & 31));
                event(v, operand_events(nd > 1, false, has(after, v), dup, false, &flags));
                opflags[o - po.o0 + lane] = (uint8_t)flags;
            }
            __syncwarp();
        }
        for (uint32_t o = o0 + lane; o < r0; o += 32) {
            const uint32_t v = q.op_vreg[o];
            uint32_t flags;
            event(v, operand_events(nd > 1, true, has(after, v), false, has(reads, v), &flags));
            opflags[o - po.o0] = (uint8_t)flags;
        }
        __syncwarp();
        int change = 0;  // of the live count, going backwards
        if (live) {
            for (uint32_t o = o0 + lane; o < r0; o += 32) {
                const uint32_t v = q.op_vreg[o];
                if (has(live, v)) { --change; atomicAnd(const_cast<uint32_t *>(live) + (v >> 5), ~(1u << (v & 31))); }
            }
            __syncwarp();
            for (uint32_t o = r0 + lane; o < o1; o += 32) {
                const uint32_t v = q.op_vreg[o], bit = 1u << (v & 31);
                if (!(atomicOr(const_cast<uint32_t *>(live) + (v >> 5), bit) & bit)) ++change;
            }
        }
        for (uint32_t o = r0 + lane; o < o1; o += 32) reads[q.op_vreg[o] >> 5] = 0;
        n_ev = __reduce_add_sync(0xffffffffu, n_ev);
        change = __reduce_add_sync(0xffffffffu, change);
        if (lane == 0) { s_ev[k] = n_ev; s_d[k] = change; }
        __syncwarp();
    }
}

// ============================================================================ k_count
// One thread block per chunk.  First the live set after the last instruction of every piece (one thread per
// bitset word, backwards over the chunk's pieces).  Then one warp per piece, one lane per operand (count_narrow): the operand
// flags, the walk events and the change of the live count of every instruction follow without a serial walk; and the set of
// vregs whose occupancy changes inside the block.  Last, offsets inside the chunk.  WIDE: some piece of the launch has more
// than PIECE_OPERANDS operands.
template <int N, bool WIDE>
__global__ void __launch_bounds__(PC_NT) k_count(const __grid_constant__ LiveMany<N> a)
{
    LIVE_ARGS;
    __shared__ uint32_t s_scan[34], s_ev[PC_WARPS][PIECE_INSTRS];
    __shared__ int s_d[PC_WARPS][PIECE_INSTRS];
    const uint32_t c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (c >= q.nC) return;
    const uint32_t p0 = q.chunk_piece_off[c], p1 = q.chunk_piece_off[c + 1];
    const uint32_t blk = q.chunk_blk[c];
    uint32_t *touch = q.blk_touch + (size_t)blk * q.Wv;
    Piece po;
    uint32_t x = 0;  // the operands of the warp's (first) piece
    if (p0 + warp < p1) {
        po.init(q, p0 + warp);
        x = po.get(q, lane);
    }
    pdl_go();
    pdl_wait();
    for (uint32_t w = tid; w < q.Wv; w += PC_NT) {
        uint32_t live = q.chunk_end[(size_t)c * q.Wv + w];
        for (uint32_t pe = p1; pe > p0;) {
            uint32_t pu[8], pd[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool ok = pe - p0 > (uint32_t)j;
                pu[j] = ok ? q.piece_use[(size_t)(pe - 1 - j) * q.Wv + w] : 0u;
                pd[j] = ok ? q.piece_def[(size_t)(pe - 1 - j) * q.Wv + w] : 0u;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (pe - p0 > (uint32_t)j) {
                    q.piece_end[(size_t)(pe - 1 - j) * q.Wv + w] = live;
                    live = pu[j] | (live & ~pd[j]);
                }
            pe -= min(pe - p0, 8u);
        }
    }
    __syncthreads();
    for (uint32_t p = p0 + warp; p < p1; p += PC_WARPS) {
        const uint32_t *end = q.piece_end + (size_t)p * q.Wv;
        if (p != p0 + warp) {
            po.init(q, p);
            x = po.get(q, lane);
        }
        const uint32_t touched = lane < po.n ? __ldcg(&touch[po_vreg(x) >> 5]) : 0u;
        uint32_t cnt = 0;
        for (uint32_t w = lane; w < q.Wv; w += 32) cnt += __popc(end[w]);
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (!WIDE || po.n <= PIECE_OPERANDS) {
            count_narrow(po, x, end, q.opflags + po.o0, touch, touched, s_d[warp], s_ev[warp]);
        } else {  // the sets of reads and of what is live: in shared memory if they fit, else in the rows of the piece's own sets, used up by now
            extern __shared__ uint32_t sm[];
            uint32_t *reads = q.wide_smem ? sm + (size_t)warp * 2 * q.Wv : q.piece_def + (size_t)p * q.Wv;
            uint32_t *live = q.wide_smem ? reads + q.Wv : q.piece_use + (size_t)p * q.Wv;
            for (uint32_t w = lane; w < q.Wv; w += 32) reads[w] = 0;
            __syncwarp();
            count_wide<true>(q, po, end, reads, po.ni > 1 ? live : nullptr, q.opflags + po.o0, touch, s_d[warp], s_ev[warp]);
        }
        __syncwarp();
        // live after instruction k = live after the piece + what the later instructions add going backwards
        if (lane < po.ni) {
            int live = (int)cnt;
            for (uint32_t u = lane + 1; u < po.ni; ++u) live += s_d[warp][u];
            q.lo_rel[po.i0 + lane] = (uint32_t)live;
            q.ev_rel[po.i0 + lane] = s_ev[warp][lane];
        }
        __syncwarp();
    }
    __syncthreads();
    const uint32_t i0 = q.chunk_i0[c], i1 = q.chunk_i1[c];
    unsigned long long lo_sum = 0;
    uint32_t ev_sum = 0;
    for (uint32_t ib = i0; ib < i1; ib += PC_NT) {
        const uint32_t i = ib + tid;
        const uint32_t a = i < i1 ? q.lo_rel[i] : 0u, e = i < i1 ? q.ev_rel[i] : 0u;
        uint32_t ta, te;  // (PC_NT lists of at most 65,535 entries: 32 bits hold the sum)
        const uint32_t xa = block_excl_scan(a, s_scan, &ta), xe = block_excl_scan(e, s_scan, &te);
        if (i < i1) { q.lo_rel[i] = (uint32_t)lo_sum + xa; q.ev_rel[i] = ev_sum + xe; }
        lo_sum += ta;
        ev_sum += te;
    }
    if (tid == 0) { q.chunk_lo[c] = lo_sum; q.chunk_ev[c] = ev_sum; }
}

// The live set before piece p of chunk c (p0 = the chunk's first piece), one word.
__device__ __forceinline__ uint32_t live_before(const LiveArgs &q, uint32_t c, uint32_t p, uint32_t p0, uint32_t w)
{
    return p == p0 ? q.chunk_entry[(size_t)c * q.Wv + w] : q.piece_end[(size_t)(p - 1) * q.Wv + w];
}
// The through-set of block b, one word, from what touched its vregs.
__device__ __forceinline__ uint32_t through_word(const LiveArgs &q, uint32_t b, uint32_t w)
{
    return q.use_th ? q.blk_in[(size_t)b * q.Wv + w] & ~q.blk_touch[(size_t)b * q.Wv + w] : 0u;
}

// The offsets of everything, from what the chunks, blocks and short chunks hold, by the first LV_TOTALS warps of a block: a
// warp per total, the scans side by side; a lane takes up to 8 consecutive values at a time, whose loads are in flight
// together.  GLOBAL: they lie in global memory and other blocks have written them (loads past the L1 cache).
template <bool GLOBAL>
__device__ __forceinline__ void live_offsets(const LiveArgs &q, unsigned long long *s_tot, const unsigned long long *chunk_lo,
                                             const uint32_t *centry_cnt, const uint32_t *chunk_ev, const uint32_t *th_cnt,
                                             const uint32_t *blk_off, const uint32_t *short_ev, const uint32_t *short_ent)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto load = [](const auto *p) { return GLOBAL ? __ldcg(p) : *p; };
    // Exclusive offsets of n values into dst[0..n) (null: none), dst[n] = total, clipped to 32 bits; the total is returned.
    auto offsets = [&](uint32_t n, uint32_t *dst, auto value, auto store) -> unsigned long long {
        unsigned long long carry = 0;
        for (uint32_t j0 = 0; j0 < n; j0 += 256) {
            const uint32_t j = j0 + lane * 8;
            unsigned long long x[8], sum = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = j + u < n ? value(j + u) : 0ull;
#pragma unroll
            for (int u = 0; u < 8; ++u) sum += x[u];
            unsigned long long inc = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= (uint32_t)d) inc += y;
            }
            unsigned long long at = carry + inc - sum;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (j + u < n) store(j + u, (uint32_t)at);
                at += x[u];
            }
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (dst && lane == 0) dst[n] = carry > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)carry;
        return carry;
    };
    auto into = [](uint32_t *dst) { return [dst](uint32_t j, uint32_t at) { dst[j] = at; }; };
    unsigned long long tot = 0;
    if (warp == LV_TOT_LO) {
        tot = offsets(q.nC, q.chunk_lo0, [&](uint32_t c) { return load(chunk_lo + c); }, into(q.chunk_lo0));
        if (lane == 0) q.lo_off[q.nI] = tot > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)tot;
    } else if (warp == LV_TOT_EV) {
        tot = offsets(q.nC, q.cev_off, [&](uint32_t c) -> unsigned long long {
            return (load(centry_cnt + c) + load(chunk_ev + c) + 7u) / 8u * 8u;
        }, into(q.cev_off));
    } else if (warp == LV_TOT_TH) {
        tot = offsets(q.nB, q.th_off, [&](uint32_t b) -> unsigned long long { return load(th_cnt + b); }, into(q.th_off));
    } else if (warp == LV_TOT_LS) {
        // short lists (see vl_program): what the through-sets take off the lists of the blocks before b
        tot = offsets(q.nB, nullptr, [&](uint32_t b) -> unsigned long long {
            return (unsigned long long)(blk_off[b + 1] - blk_off[b]) * load(th_cnt + b);
        }, [&](uint32_t b, uint32_t pre) { q.ls_adj[b] = pre - blk_off[b] * load(th_cnt + b); });
    } else if (warp == LV_TOT_SEV) {  // a group of 32 short chunks per round: its longest
#pragma unroll 4
        for (uint32_t g = 0; g * 32 < q.nS; ++g) {
            const uint32_t m = __reduce_max_sync(0xffffffffu, g * 32 + lane < q.nS ? load(short_ev + g * 32 + lane) : 0u);
            if (lane == 0) q.sev_off[g] = (uint32_t)tot;
            tot += m;
        }
        if (lane == 0) q.sev_off[(q.nS + 31) / 32] = (uint32_t)tot;
        tot *= 32;
    } else if (warp == LV_TOT_SEN) {
        tot = offsets(q.nS, q.sen_off, [&](uint32_t s) -> unsigned long long { return load(short_ent + s); }, into(q.sen_off));
    }
    if (warp < LV_TOTALS && lane == 0) s_tot[warp] = tot;
}
// The totals and the status word to the host (one thread).
__device__ __forceinline__ void live_totals(const LiveArgs &q, unsigned long long *s_tot, uint32_t st)
{
    s_tot[LV_TOT_LS] = s_tot[LV_TOT_LO] - s_tot[LV_TOT_LS];
    if (s_tot[LV_TOT_LO] > 0xFFFFFFF0ull) st |= ST_SIZE_OVERFLOW;
    q.host_out[0] = st;
    unsigned long long *h = reinterpret_cast<unsigned long long *>(q.host_out + 2);
    for (int j = 0; j < LV_TOTALS; ++j) h[j] = s_tot[j];
}

// ============================================================================ k_offsets
// Thread blocks [0, nC): entry events of a chunk and events of its short chunks; [nC, nC + nB): the through-set
// of a block (live on entry and never touched by an event inside it).  The block that finishes last makes the
// offsets: list entries per chunk, walk events per chunk (padded to groups of 8), through-sets per block, steps
// per 32 short chunks; and writes the totals and the status word to pinned host memory.
template <int N>
__global__ void __launch_bounds__(OFF_NT) k_offsets(const __grid_constant__ LiveMany<N> a)
{
    LIVE_ARGS;
    __shared__ uint32_t s_scan[34];
    __shared__ unsigned long long s_tot[LV_TOTALS];
    __shared__ uint32_t s_last;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (blockIdx.x >= q.nC + q.nB) return;
    pdl_go();
    pdl_wait();
    if (blockIdx.x < q.nC) {
        const uint32_t c = blockIdx.x, b = q.chunk_blk[c], p0 = q.chunk_piece_off[c];
        const uint32_t s1 = q.chunk_short_off[c + 1];
        for (uint32_t s = q.chunk_short_off[c] + warp; s < s1; s += OFF_NT / 32) {
            const uint32_t p = q.short_p0[s];
            uint32_t cnt = 0;
            for (uint32_t w = lane; w < q.Wv; w += 32) cnt += __popc(live_before(q, c, p, p0, w) & ~through_word(q, b, w));
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            if (lane == 0) {
                if (p == p0) q.centry_cnt[c] = cnt;
                const uint32_t ev1 = s + 1 < s1 ? q.ev_rel[q.piece_i0[q.short_p0[s + 1]]] : q.chunk_ev[c];
                q.short_ent[s] = cnt;
                q.short_ev[s] = ev1 - q.ev_rel[q.piece_i0[p]];
            }
        }
    } else {
        const uint32_t b = blockIdx.x - q.nC;
        uint32_t cnt = 0, total;
        for (uint32_t w = tid; w < q.Wv; w += OFF_NT) {
            const uint32_t t = through_word(q, b, w);
            q.blk_th[(size_t)b * q.Wv + w] = t;
            cnt += __popc(t);
        }
        block_excl_scan(cnt, s_scan, &total);
        if (tid == 0) q.th_cnt[b] = total;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&q.counters[0], 1u) == q.nC + q.nB - 1 ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    live_offsets<true>(q, s_tot, q.chunk_lo, q.centry_cnt, q.chunk_ev, q.th_cnt, q.blk_off, q.short_ev, q.short_ent);
    __syncthreads();
    if (tid == 0) live_totals(q, s_tot, __ldcg(q.status));
}

// ============================================================================ k_small
// k_sets, k_flow, k_count and k_offsets of a program of up to LIVE_SMALL_INSTRS instructions in one launch: a cluster of C
// thread blocks, each with a share of the chunks whose sets stay in its shared memory from phase to phase.  What bounds such
// a run is not work but the chain of launches and L2 round trips: 100 rows of 2,000 instructions, liveness included, 54 us
// with the four kernels, 37 with this one; of 64 instructions 38 and 28.  What the blocks need of each other (chunk sets,
// touched vregs, counts) they store into each other's shared memory, behind three cluster barriers; the fixed point over the
// blocks is cheap enough for every thread block to do all of it, which saves a barrier.  One block does the last scans.

// Composes the sets of units [j0, j1) (rows of Wv words, one word), going forwards: read before written, written.  Eight
// loads in flight.
__device__ __forceinline__ void compose_sets(const uint32_t *use, const uint32_t *def, uint32_t j0, uint32_t j1, uint32_t Wv, uint32_t &u, uint32_t &d)
{
    u = d = 0;
#pragma unroll 1
    for (; j0 < j1; j0 += 8) {
        uint32_t x[8], y[8];
#pragma unroll
        for (uint32_t t = 0; t < 8; ++t) {
            const uint32_t at = min(j0 + t, j1 - 1) * Wv;  // (once more the last one: no harm)
            x[t] = use[at];
            y[t] = def[at];
        }
#pragma unroll
        for (uint32_t t = 0; t < 8; ++t) { u |= x[t] & ~d; d |= y[t]; }
    }
}
// Live sets of units [j0, j1) going backwards from `live`: use becomes what is live after the unit, or (BEFORE) before it.
template <bool BEFORE>
__device__ __forceinline__ void live_sets(uint32_t *use, const uint32_t *def, uint32_t j0, uint32_t j1, uint32_t Wv, uint32_t live)
{
#pragma unroll 1
    for (; j1 > j0; j1 -= min(j1 - j0, 8u)) {
        uint32_t x[8], y[8];
#pragma unroll
        for (uint32_t t = 0; t < 8; ++t) {
            const uint32_t at = (j1 - 1 - min(t, j1 - j0 - 1)) * Wv;
            x[t] = use[at];
            y[t] = def[at];
        }
#pragma unroll
        for (uint32_t t = 0; t < 8; ++t) {
            if (t >= j1 - j0) break;
            if (!BEFORE) use[(j1 - 1 - t) * Wv] = live;
            live = x[t] | (live & ~y[t]);
            if (BEFORE) use[(j1 - 1 - t) * Wv] = live;
        }
    }
}

template <int N, int C>
__global__ void __launch_bounds__(SMALL_NT, 2) k_small(const __grid_constant__ LiveMany<N> a)
{
    LIVE_ARGS;
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ uint32_t s_ev[SMALL_WARPS][PIECE_INSTRS];
    __shared__ int s_d[SMALL_WARPS][PIECE_INSTRS];
    __shared__ uint32_t s_st;
    __shared__ unsigned long long s_tot[LV_TOTALS];
    namespace cg = cooperative_groups;
    const uint32_t rank = C == 1 ? 0u : blockIdx.x;  // (a grid of C blocks per program, clusters of C)
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, Wv = q.Wv;
    const uint4 *share = q.share + (C == 1 ? SMALL_BLOCKS + 1 : 0);  // first chunk, piece, instruction, operand
    const uint4 s0 = share[rank], s1 = share[rank + 1];
    const SmallSmem &L = q.small;
    uint32_t *pu = sm + L.pu, *pd = sm + L.pd, *cu = sm + L.cu, *cd = sm + L.cd, *bu = sm + L.bu, *bd = sm + L.bd, *bi = sm + L.bi,
             *bo = sm + L.bo, *bt = sm + L.bt, *piece_chunk = sm + L.pc;
    const uint32_t *blk_chunk = sm + L.blk_chunk, *chunk_piece = sm + L.chunk_piece, *chunk_blk = sm + L.chunk_blk,
                   *chunk_short = sm + L.chunk_short, *short_piece = sm + L.short_piece, *short_chunk = sm + L.short_chunk,
                   *s_so = sm + L.succ_off, *s_su = sm + L.succ;
    uint8_t *s_fl = reinterpret_cast<uint8_t *>(sm + L.fl);
    unsigned long long *s_clo = reinterpret_cast<unsigned long long *>(sm + L.clo);
    auto sync = [&] {
        if (C == 1) __syncthreads();
        else cg::this_cluster().sync();
    };
    // p of this block as block r of the cluster has it
    auto of = [&](auto *p, uint32_t r) { return C == 1 ? p : cg::this_cluster().map_shared_rank(p, r); };

    // ---- what the phases read of the program and its layout comes to shared memory, in two L2 round trips with the shares
    for (uint32_t i = tid; i < L.tab_words; i += SMALL_NT) sm[L.tab + i] = q.small_tab[i];
    const uint32_t c0 = s0.x, c1 = s1.x, p0 = s0.y, np = s1.y - s0.y, o_first = s0.w, n_ops = s1.w - s0.w;
    for (uint32_t i = tid; i <= np; i += SMALL_NT) {
        sm[L.pi + i] = q.piece_i0[p0 + i];
        sm[L.po + i] = q.piece_o0[p0 + i];
        if (i < np) piece_chunk[i] = q.piece_chunk[p0 + i];
    }
    for (uint32_t i = tid; i < n_ops; i += SMALL_NT) sm[L.xs + i] = q.op_word[o_first + i];
    for (uint32_t i = tid; i < np * Wv; i += SMALL_NT) pu[i] = pd[i] = 0;
    for (uint32_t i = tid; i < q.nB * Wv; i += SMALL_NT) bt[i] = bi[i] = 0;
    if (tid == 0) s_st = 0;
    __syncthreads();
    auto piece = [&](uint32_t j) {
        Piece x;
        x.i0 = sm[L.pi + j];
        x.ni = sm[L.pi + j + 1] - x.i0;
        x.o0 = sm[L.po + j];
        x.n = sm[L.po + j + 1] - x.o0;
        return x;
    };
    auto operand = [&](const Piece &x) { return lane < x.n ? sm[L.xs + x.o0 - o_first + lane] : 0u; };
    // ---- read and write sets of the pieces
    for (uint32_t j = warp; j < np; j += SMALL_WARPS) {
        const Piece x = piece(j);
        piece_sets(q, x, operand(x), lane, pu + j * Wv, pd + j * Wv);
    }
    sync();  // (every block has begun: its shared memory may be written to)
    // ---- the chunks', to every block
    for (uint32_t i = tid; i < (c1 - c0) * Wv; i += SMALL_NT) {
        const uint32_t c = c0 + i / Wv, w = i % Wv;
        uint32_t u, d;
        compose_sets(pu + w, pd + w, chunk_piece[c] - p0, chunk_piece[c + 1] - p0, Wv, u, d);
        for (uint32_t r = 0; r < C; ++r) {
            of(cu, r)[c * Wv + w] = u;
            of(cd, r)[c * Wv + w] = d;
        }
    }
    sync();
    // ---- block sets, fixed point, live sets at the chunk boundaries (every block: all of them)
    for (uint32_t i = tid; i < q.nB * Wv; i += SMALL_NT) {
        const uint32_t b = i / Wv, w = i % Wv;
        compose_sets(cu + w, cd + w, blk_chunk[b], blk_chunk[b + 1], Wv, bu[i], bd[i]);
    }
    __syncthreads();
    if (warp * 32 < Wv) {  // a warp per 32 words (and more of them where there are more words than lanes)
        uint32_t st = 0;
        for (uint32_t w0 = warp * 32; w0 < Wv; w0 += SMALL_NT) {
            const uint32_t w = min(w0 + lane, Wv - 1);  // (lanes past the last word do it once more)
            bool changed = true;
            for (uint32_t sweep = 0; sweep < q.nB + 2 && __any_sync(0xffffffffu, changed); ++sweep) {
                changed = false;
                uint32_t e = s_so[q.nB];
                for (uint32_t b = q.nB; b-- > 0;) {
                    const uint32_t u = bu[b * Wv + w], d = bd[b * Wv + w], was = bi[b * Wv + w], e0 = s_so[b];
                    uint32_t o = 0;
                    while (e > e0) o |= bi[s_su[--e] * Wv + w];
                    const uint32_t i = u | (o & ~d);
                    changed |= i != was;
                    bi[b * Wv + w] = i;
                    bo[b * Wv + w] = o;
                }
            }
            if (changed) st |= ST_NO_CONVERGE;
            if (bi[w] != 0) st |= ST_NOT_STRICT;  // block 0 is the entry
        }
        st = __reduce_or_sync(0xffffffffu, st);
        if (st && lane == 0) atomicOr(&s_st, st);
    }
    __syncthreads();
    for (uint32_t i = tid; i < q.nB * Wv; i += SMALL_NT) {
        const uint32_t b = i / Wv, w = i % Wv;
        live_sets<true>(cu + w, cd + w, blk_chunk[b], blk_chunk[b + 1], Wv, bo[i]);
    }
    __syncthreads();
    // ---- live sets behind the pieces of the share
    for (uint32_t i = tid; i < (c1 - c0) * Wv; i += SMALL_NT) {
        const uint32_t c = c0 + i / Wv, w = i % Wv, b = chunk_blk[c];
        const uint32_t live = c + 1 < blk_chunk[b + 1] ? cu[(c + 1) * Wv + w] : bo[b * Wv + w];
        live_sets<false>(pu + w, pd + w, chunk_piece[c] - p0, chunk_piece[c + 1] - p0, Wv, live);
    }
    __syncthreads();
    // ---- operand flags, touched vregs, events and live counts (see k_count); offsets inside the pieces
    for (uint32_t j = warp; j < np; j += SMALL_WARPS) {
        const uint32_t *end = pu + j * Wv;
        uint32_t *touch = bt + chunk_blk[piece_chunk[j]] * Wv;
        const Piece x = piece(j);
        uint32_t cnt = 0;
        for (uint32_t w = lane; w < Wv; w += 32) cnt += __popc(end[w]);
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (x.n <= PIECE_OPERANDS) {
            count_narrow(x, operand(x), end, s_fl + x.o0 - o_first, touch, 0u, s_d[warp], s_ev[warp]);
        } else {
            uint32_t *reads = sm + L.rd + warp * Wv;
            for (uint32_t w = lane; w < Wv; w += 32) reads[w] = 0;
            __syncwarp();
            count_wide<false>(q, x, end, reads, nullptr, s_fl + x.o0 - o_first, touch, s_d[warp], s_ev[warp]);
        }
        __syncwarp();
        // live after instruction k = live after the piece + what the later instructions add going backwards
        const bool mine = lane < x.ni;
        int later = mine && lane + 1 < x.ni ? s_d[warp][lane + 1] : 0;
#pragma unroll
        for (int d = 1; d < PIECE_INSTRS; d <<= 1) later += __shfl_down_sync(0xffffffffu, later, d);  // (zeros beyond the piece)
        const uint32_t lo = mine ? (uint32_t)((int)cnt + later) : 0u, ev = mine ? s_ev[warp][lane] : 0u;
        uint32_t lo_i = lo, ev_i = ev;
#pragma unroll
        for (int d = 1; d < PIECE_INSTRS; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, lo_i, d), z = __shfl_up_sync(0xffffffffu, ev_i, d);
            if (lane >= (uint32_t)d) { lo_i += y; ev_i += z; }
        }
        if (mine) { sm[L.lo + j * PIECE_INSTRS + lane] = lo_i - lo; sm[L.ev + j * PIECE_INSTRS + lane] = ev_i - ev; }
        if (lane == PIECE_INSTRS - 1) { sm[L.plo + j] = lo_i; sm[L.pev + j] = ev_i; }
        __syncwarp();
    }
    __syncthreads();
    // ---- touched vregs to every block; offsets inside the chunks (a warp per chunk, a lane per piece), events of the short chunks
    if (C > 1)
        for (uint32_t i = tid; i < q.nB * Wv; i += SMALL_NT) {
            const uint32_t t = bt[i];  // (bits that other blocks have stored meanwhile go round once more: no harm)
            if (t)
                for (uint32_t r = 0; r < C; ++r)
                    if (r != rank) atomicOr(of(bt, r) + i, t);
        }
    uint32_t *cev = of(sm + L.cev, 0), *cent = of(sm + L.cent, 0), *sent = of(sm + L.sent, 0), *sev = of(sm + L.sev, 0);
    unsigned long long *clo = of(s_clo, 0);
    for (uint32_t c = c0 + warp; c < c1; c += SMALL_WARPS) {
        const uint32_t first = chunk_piece[c] - p0, last = chunk_piece[c + 1] - p0;
        unsigned long long lo_sum = 0;
        uint32_t ev_sum = 0;
        for (uint32_t j0 = first; j0 < last; j0 += 32) {
            const uint32_t j = j0 + lane;
            const uint32_t x = j < last ? sm[L.plo + j] : 0u, y = j < last ? sm[L.pev + j] : 0u;
            uint32_t xi = x, yi = y;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t xo = __shfl_up_sync(0xffffffffu, xi, d), yo = __shfl_up_sync(0xffffffffu, yi, d);
                if (lane >= (uint32_t)d) { xi += xo; yi += yo; }
            }
            if (j < last) { sm[L.plo + j] = (uint32_t)lo_sum + xi - x; sm[L.pev + j] = ev_sum + yi - y; }
            lo_sum += __shfl_sync(0xffffffffu, xi, 31);
            ev_sum += __shfl_sync(0xffffffffu, yi, 31);
        }
        __syncwarp();
        if (lane == 0) { clo[c] = lo_sum; cev[c] = ev_sum; sm[L.cev + c] = ev_sum; }
        const uint32_t s_hi = chunk_short[c + 1];
        for (uint32_t s = chunk_short[c] + lane; s < s_hi; s += 32) {
            const uint32_t e0 = sm[L.pev + short_piece[s] - p0], e1 = s + 1 < s_hi ? sm[L.pev + short_piece[s + 1] - p0] : ev_sum;
            sev[s] = sm[L.sev + s] = e1 - e0;
        }
    }
    sync();
    // ---- through-sets (every block: all of them), what is occupied when chunks and short chunks of the share begin
    for (uint32_t i = tid; i < q.nB * Wv; i += SMALL_NT) bu[i] = q.use_th ? bi[i] & ~bt[i] : 0u;
    __syncthreads();
    for (uint32_t s = chunk_short[c0] + warp; s < chunk_short[c1]; s += SMALL_WARPS) {
        const uint32_t p = short_piece[s], c = short_chunk[s];
        const bool first = p == chunk_piece[c];
        const uint32_t *live = first ? cu + c * Wv : pu + (p - 1 - p0) * Wv, *t = bu + chunk_blk[c] * Wv;
        uint32_t cnt = 0;
        for (uint32_t w = lane; w < Wv; w += 32) cnt += __popc(live[w] & ~t[w]);
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) {
            sent[s] = cnt;
            if (first) cent[c] = sm[L.cent + c] = cnt;
        }
    }
    if (rank == 0)
        for (uint32_t b = warp; b < q.nB; b += SMALL_WARPS) {
            uint32_t cnt = 0;
            for (uint32_t w = lane; w < Wv; w += 32) cnt += __popc(bu[b * Wv + w]);
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            if (lane == 0) sm[L.thn + b] = cnt;
        }
    sync();
    // ---- everything to global memory (stores in front of a cluster barrier would be waited for there); the offsets
    pdl_go();
    pdl_wait();  // an earlier call's kernels may still read what is written from here on
    if (rank == 0) {
        live_offsets<false>(q, s_tot, s_clo, sm + L.cent, sm + L.cev, sm + L.thn, sm + L.blk_off, sm + L.sev, sm + L.sent);
        for (uint32_t i = tid; i < q.nB * Wv; i += SMALL_NT) { q.blk_in[i] = bi[i]; q.blk_out[i] = bo[i]; q.blk_th[i] = bu[i]; }
        for (uint32_t b = tid; b < q.nB; b += SMALL_NT) { q.el_count[b] = 0; q.th_cnt[b] = sm[L.thn + b]; }
    }
    for (uint32_t i = tid; i < n_ops; i += SMALL_NT) q.opflags[o_first + i] = s_fl[i];
    for (uint32_t i = tid; i < np * Wv; i += SMALL_NT) q.piece_end[(size_t)p0 * Wv + i] = pu[i];
    for (uint32_t i = tid; i < (c1 - c0) * Wv; i += SMALL_NT) q.chunk_entry[(size_t)c0 * Wv + i] = cu[c0 * Wv + i];
    for (uint32_t c = c0 + tid; c < c1; c += SMALL_NT) { q.chunk_ev[c] = sm[L.cev + c]; q.centry_cnt[c] = sm[L.cent + c]; }
    for (uint32_t s = chunk_short[c0] + tid; s < chunk_short[c1]; s += SMALL_NT) q.short_ev[s] = sm[L.sev + s];
    for (uint32_t i = tid; i < np * PIECE_INSTRS; i += SMALL_NT) {
        const uint32_t j = i / PIECE_INSTRS, k = sm[L.pi + j] + i % PIECE_INSTRS;
        if (k >= sm[L.pi + j + 1]) continue;
        q.lo_rel[k] = sm[L.plo + j] + sm[L.lo + i];
        q.ev_rel[k] = sm[L.pev + j] + sm[L.ev + i];
    }
    if (rank) return;
    __syncthreads();
    if (tid == 0) {
        const uint32_t st = s_st;
        *q.status = st;
        live_totals(q, s_tot, st);
    }
}

// The operand words of a layout's pieces (see Piece), a warp per piece.
__global__ void __launch_bounds__(NT) k_operand_words(uint32_t nP, const uint32_t *__restrict__ piece_i0, const uint32_t *__restrict__ op_off,
                                                      const uint8_t *__restrict__ ndefs, const uint32_t *__restrict__ op_vreg, uint32_t *op_word)
{
    const uint32_t p = blockIdx.x * (NT / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (p >= nP) return;
    const uint32_t i0 = piece_i0[p], i1 = piece_i0[p + 1], o0 = op_off[i0], n = op_off[i1] - o0;
    if (n > PIECE_OPERANDS) {
        for (uint32_t j = lane, i = i0; j < n; j += 32) {
            while (op_off[i + 1] <= o0 + j) ++i;
            const uint32_t v = op_vreg[o0 + j];
            bool fresh = true;  // no earlier instruction of the piece writes the vreg
            for (uint32_t h = i0; h < i; ++h)
                for (uint32_t d = 0; d < ndefs[h]; ++d) fresh = fresh && op_vreg[op_off[h] + d] != v;
            op_word[o0 + j] = v | ((i - i0) << 16) | (o0 + j - op_off[i] < ndefs[i] ? OW_DEF : (fresh ? OW_EXPOSED : 0u));
        }
        return;
    }
    const bool mine = lane < n;
    uint32_t x = 0;
    if (mine) {
        uint32_t i = i0;
        while (op_off[i + 1] <= o0 + lane) ++i;
        x = op_vreg[o0 + lane] | ((i - i0) << 16) | (o0 + lane - op_off[i] < ndefs[i] ? OW_DEF : 0u) | (ndefs[i] > 1 ? OW_MANY : 0u);
    }
    const uint32_t here = same_instr(x, mine), same = __match_any_sync(0xffffffffu, mine ? po_vreg(x) : 0x10000u + lane);
    const uint32_t defs = __ballot_sync(0xffffffffu, mine && po_def(x));
    const uint32_t before = mine ? low_bits(__ffs(here) - 1) : 0u, later = mine ? same & ~(before | here) : 0u;
    const uint32_t here_next = __shfl_sync(0xffffffffu, here, later ? __ffs(later) - 1 : 0);
    if (!mine) return;
    if (!po_def(x) && (same & here & ~defs & low_bits(lane))) x |= OW_DUP;
    if (same & here & (po_def(x) ? ~defs : defs)) x |= OW_OTHER;
    if (!po_def(x) && !(same & before & defs)) x |= OW_EXPOSED;
    if (later) x |= OW_LATER | (same & here_next & ~defs ? OW_READ : 0u);
    op_word[o0 + lane] = x;
}

// First occurrence and first definition of every vreg.
__global__ void k_first_occ(uint32_t nI, const uint32_t *__restrict__ op_off, const uint8_t *__restrict__ ndefs,
                            const uint32_t *__restrict__ op_vreg, uint32_t *first_occ, uint32_t *first_def_instr)
{
    const uint32_t i = blockIdx.x * NT + threadIdx.x;
    if (i >= nI) return;
    const uint32_t o0 = op_off[i], o1 = op_off[i + 1], nd = ndefs[i];
    for (uint32_t o = o0; o < o1; ++o) {
        atomicMin(&first_occ[op_vreg[o]], o);
        if (o < o0 + nd) atomicMin(&first_def_instr[op_vreg[o]], i);
    }
}

__global__ void k_vreg_info(uint32_t V, const uint8_t *__restrict__ width, const uint32_t *__restrict__ first_occ,
                            const uint32_t *__restrict__ first_def_instr, uint32_t *vinfo)
{
    const uint32_t v = blockIdx.x * NT + threadIdx.x;
    if (v >= V) return;
    vinfo[v] = width[v] | (first_occ[v] != 0xFFFFFFFFu ? VINFO_OCCURS : 0u) |
               (first_def_instr[v] != 0xFFFFFFFFu ? VINFO_DEFINED : 0u);
}

// Vreg id per operand (16 bit), a byte of first-occurrence bits per 8 operands, and the operand metadata of the eight-candidate
// table kernel, per four operands: the byte offsets of the vregs' 16-byte table entries and a nibble of first-occurrence bits;
// there, operands beyond n_operands (the arrays are padded to whole tiles) name the spare entry V and are never a first
// occurrence.  One thread per 8 operands of the padded arrays.
__global__ void k_operand_tables(uint32_t nO, uint32_t nOp8, uint32_t n_padded, uint32_t V, const uint32_t *__restrict__ op_vreg,
                                 const uint32_t *__restrict__ first_occ, uint16_t *vreg16, uint8_t *first8, uint4 *opoff, uint8_t *first4)
{
    const uint32_t s = blockIdx.x * NT + threadIdx.x;
    if (s >= n_padded) return;
    uint32_t off[8], f = 0, padding = 0;
    for (uint32_t j = 0; j < 8; ++j) {
        const uint32_t o = s * 8 + j, v = o < nO ? op_vreg[o] : V;
        off[j] = v * 16u;
        if (o < nO) f |= (first_occ[v] == o ? 1u : 0u) << j;
        else padding |= 1u << j;  // a padding operand writes the spare table entry and is never compared
        if (o < nOp8) vreg16[o] = (uint16_t)v;
    }
    if (s < nOp8 / 8) first8[s] = (uint8_t)(f | padding);
    opoff[2 * s] = make_uint4(off[0], off[1], off[2], off[3]);
    opoff[2 * s + 1] = make_uint4(off[4], off[5], off[6], off[7]);
    first4[2 * s] = (uint8_t)(f & 15u);
    first4[2 * s + 1] = (uint8_t)(f >> 4);
}

// Walk events are stored in groups of 8, 112 bytes per group, field by field so that the walk
// fetches a group with 16-byte loads: off[8] (32 bit: byte offset of the vreg's row in a table of
// 64 16-bit entries per vreg), toggle[8] (32 bit: the width-w mask (1<<w)-1, or 0), test[8]
// (likewise), wl[8] (16 bit: 32 - width; the range straddles a 32-bit word iff
// (register & 31) > wl).  Ranges wider than 32 registers carry wl = 0x8000 | width and
// toggle, test as 0/1 flags.  A no-op names the spare vreg V with empty masks.
// And once more in 4 bytes for k_eight, where it takes the program: EV8_* (vl_internal.cuh).
__device__ __forceinline__ void put_event(const LiveArgs &q, size_t idx, uint32_t v, uint32_t w, bool test, bool toggle)
{
    unsigned char *g = reinterpret_cast<unsigned char *>(q.ev) + (idx >> 3) * 112;
    const uint32_t slot = (uint32_t)(idx & 7);
    const uint32_t wm = w > 32 ? 1u : (w == 32 ? 0xFFFFFFFFu : ((1u << w) - 1u));
    reinterpret_cast<uint32_t *>(g)[slot] = v * 128u;
    reinterpret_cast<uint32_t *>(g + 32)[slot] = toggle ? wm : 0u;
    reinterpret_cast<uint32_t *>(g + 64)[slot] = test ? wm : 0u;
    reinterpret_cast<uint16_t *>(g + 96)[slot] = (uint16_t)(w > 32 ? (0x8000u | w) : (32u - w));
    if (q.ev8) q.ev8[idx] = v * 16u | (test ? EV8_TEST : 0u) | (toggle ? 0u : EV8_HOLD) | (test || toggle ? wm << EV8_MASK_SHIFT : 0u);
}

// ============================================================================ k_fill
// Four kinds of thread blocks in one grid: [0, ceil(nP / LV_WARPS)) live-after lists, a warp per piece; then nC
// blocks with the walk events of a chunk; then the blocks with the events of short chunks, a warp per
// short chunk; then nB blocks with the through-set list of a block.

// Appends the set bits of word(w), w = 0 .. Wv - 1, in ascending order: emit(rank, bit index).  One warp.
// Returns the number of bits.
template <class W, class F>
__device__ __forceinline__ uint32_t warp_bits(uint32_t Wv, uint32_t lane, W word, F emit)
{
    uint32_t at = 0;
    for (uint32_t w0 = 0; w0 < Wv; w0 += 32) {
        uint32_t x = w0 + lane < Wv ? word(w0 + lane) : 0u;
        const uint32_t n = __popc(x);
        uint32_t inc = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
            if (lane >= (uint32_t)d) inc += y;
        }
        uint32_t rank = at + inc - n;
        while (x) {
            emit(rank++, (w0 + lane) * 32 + __ffs(x) - 1);
            x &= x - 1;
        }
        at += __shfl_sync(0xffffffffu, inc, 31);
    }
    return at;
}

// The walk events of instruction i in order: the releases of dying reads, the definitions, the releases of dead
// co-definitions: put(index, vreg, test, toggle).  skip(operand) is called for definitions without an event.
template <class F, class G>
__device__ __forceinline__ void instr_events(const LiveArgs &q, uint32_t i, F put, G skip)
{
    const uint32_t o0 = q.op_off[i], o1 = q.op_off[i + 1], nd = q.ndefs[i];
    uint32_t e = 0;
    for (uint32_t o = o0 + nd; o < o1; ++o)
        if (q.opflags[o] & OPF_KILL) put(e++, q.op_vreg[o], false, true);
    for (uint32_t o = o0; o < o0 + nd; ++o) {
        const uint32_t f = q.opflags[o];
        if (f & OPF_ELIDE) skip(o);
        else put(e++, q.op_vreg[o], true, (f & OPF_SET) != 0);
    }
    if (nd > 1)
        for (uint32_t o = o0; o < o0 + nd; ++o)
            if ((q.opflags[o] & OPF_POST) && !(q.opflags[o] & OPF_ELIDE)) put(e++, q.op_vreg[o], false, true);
}

template <int N>
__global__ void __launch_bounds__(LV_NT) k_fill(const __grid_constant__ LiveMany<N> a)
{
    LIVE_ARGS;
    extern __shared__ uint32_t sm[];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t role = blockIdx.x;
    pdl_go();
    const uint32_t n_list = (q.nP + LV_WARPS - 1) / LV_WARPS, n_short = ((q.nS + 31) & ~31u) / LV_WARPS;
    if (role < n_list) {
        // Two lists per instruction: the vregs live after it, ascending, and the same without the block's through-set (every
        // instruction of the block has all of that in its live-after set, so the short list of instruction i starts at
        // lo_off[i] - ls_adj[b] - i * th_cnt[b]).  The lists of a piece's eight instructions differ by what the piece
        // touches: its members (live after the piece, or an operand) are found once, each with a mask of the
        // instructions it is live after, and a ballot per instruction gives 32 members their places in its two lists.
        // (Walking the bitset word by word for every instruction, 48 programs of 2,500 instructions took 67.5 us, 52.6
        // now; one of 32,000 73 and 52.)
        const uint32_t p = role * LV_WARPS + warp;
        const bool mine = p < q.nP;
        const uint32_t c = mine ? q.piece_chunk[p] : 0u, b = mine ? q.chunk_blk[c] : 0u;
        Piece po{};
        uint32_t x0 = 0;  // the first 32 operands (all of them, as a rule)
        uint32_t o_k = 0, nd_k = 0, n_reads = 0;  // lane k: first operand, definitions and reads of instruction k
        if (mine) {
            po.init(q, p);
            x0 = po.get(q, lane);
            if (lane < po.ni) {
                o_k = q.op_off[po.i0 + lane];
                nd_k = q.ndefs[po.i0 + lane];
                n_reads = q.op_off[po.i0 + lane + 1] - o_k - nd_k;
            }
        }
        uint32_t v0 = q.V;  // and its first defined vreg
        if (nd_k) v0 = q.op_vreg[o_k];
        pdl_wait();
        if (!mine) return;
        uint32_t *s_end = sm + (size_t)warp * (2 * q.Wv + FILL_WARP_WORDS), *s_u = s_end + q.Wv, *s_rank = s_u + q.Wv, *s_mem = s_rank + 32;
        uint8_t *s_flag = reinterpret_cast<uint8_t *>(s_mem + 1024);
        const uint32_t *th = q.blk_th + (size_t)b * q.Wv;
        const uint32_t ls_sub = q.ls_adj[b], ls_mul = q.th_cnt[b];
        const uint32_t i0 = po.i0;
        uint32_t my_lo = 0;
        if (lane < po.ni) my_lo = q.chunk_lo0[c] + q.lo_rel[i0 + lane];
        const uint32_t th0 = nd_k ? (th[v0 >> 5] >> (v0 & 31)) & 1u : 0u;  // whether that vreg is in the through-set
        for (uint32_t w = lane; w < q.Wv; w += 32) s_end[w] = s_u[w] = q.piece_end[(size_t)p * q.Wv + w];
        if (lane < po.ni) q.lo_off[i0 + lane] = my_lo;
        __syncwarp();
        for (uint32_t r = 0; r < po.n; r += 32) {
            const uint32_t x = r == 0 ? x0 : po.get(q, r + lane);
            if (r + lane < po.n) atomicOr(&s_u[po_vreg(x) >> 5], 1u << (x & 31));
        }
        __syncwarp();
        uint32_t at[PIECE_INSTRS], as[PIECE_INSTRS];  // where the lists of instruction k go on
#pragma unroll
        for (uint32_t k = 0; k < PIECE_INSTRS; ++k) {
            at[k] = __shfl_sync(0xffffffffu, my_lo, k);
            as[k] = at[k] - ls_sub - (i0 + k) * ls_mul;
        }
        const uint32_t below = low_bits(lane), is_instr = 0xFFu & ~low_bits(PIECE_INSTRS - po.ni);  // bit 7 - k: instruction k
        for (uint32_t w0 = 0; w0 < q.Wv; w0 += 32) {  // (at most 1,024 members at a time)
            const uint32_t w = w0 + lane;
            const uint32_t u = w < q.Wv ? s_u[w] : 0u, e = w < q.Wv ? s_end[w] : 0u, t = w < q.Wv ? th[w] : 0u;
            if (!__any_sync(0xffffffffu, u != 0)) continue;
            const uint32_t n_own = __popc(u);
            uint32_t inc = n_own;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
                if (lane >= (uint32_t)d) inc += y;
            }
            const uint32_t rank0 = inc - n_own, n_mem = __shfl_sync(0xffffffffu, inc, 31);
            s_rank[lane] = rank0;
            // every lane lists its own word, or the warp word by word, whichever is shorter
            uint32_t words = __ballot_sync(0xffffffffu, u != 0);
            if (__reduce_max_sync(0xffffffffu, n_own) <= 2 * __popc(words)) {
                uint32_t rest = u, rank = rank0;
                for (; rest; rest &= rest - 1, ++rank) {
                    const uint32_t j = __ffs(rest) - 1;
                    s_mem[rank] = w * 32 + j;
                    s_flag[rank] = (uint8_t)(((e >> j) & 1u) | (((t >> j) & 1u) << 1));
                }
            } else {
                for (; words; words &= words - 1) {
                    const uint32_t src = __ffs(words) - 1;
                    const uint32_t us = __shfl_sync(0xffffffffu, u, src), es = __shfl_sync(0xffffffffu, e, src);
                    const uint32_t ts = __shfl_sync(0xffffffffu, t, src), rank = __shfl_sync(0xffffffffu, rank0, src) + __popc(us & below);
                    if ((us >> lane) & 1u) {
                        s_mem[rank] = (w0 + src) * 32 + lane;
                        s_flag[rank] = (uint8_t)(((es >> lane) & 1u) | (((ts >> lane) & 1u) << 1));
                    }
                }
            }
            __syncwarp();
            for (uint32_t r = 0; r < po.n; r += 32) {  // bits 16 + 7 - k, 24 + 7 - k: instruction k reads, defines the member
                const uint32_t x = r == 0 ? x0 : po.get(q, r + lane), v = po_vreg(x);
                if (r + lane < po.n && v >> 10 == w0 >> 5)
                    atomicOr(&s_mem[s_rank[(v >> 5) & 31] + __popc(s_u[v >> 5] & low_bits(v & 31))],
                             1u << ((po_def(x) ? 31u : 23u) - po_instr(x)));
            }
            __syncwarp();
            for (uint32_t m0 = 0; m0 < n_mem; m0 += 32) {
                const bool ok = m0 + lane < n_mem;
                const uint32_t x = ok ? s_mem[m0 + lane] : 0u, flag = ok ? s_flag[m0 + lane] : 0u;
                // live after instruction k iff the next instruction that touches the member reads it (in the piece's last
                // stretch: iff it is live after the piece).  That is a carry that a read generates and a definition stops,
                // from the last instruction to the first: an addition.
                const uint32_t rd = (x >> 16) & 0xFFu, pass = (~(x >> 24) & 0xFFu) | rd;
                const uint32_t mask = ok ? (rd ^ pass ^ (rd + pass + (flag & 1u))) & is_instr : 0u;
                const uint32_t short_lanes = ~__ballot_sync(0xffffffffu, flag & 2u);
#pragma unroll
                for (uint32_t k = 0; k < PIECE_INSTRS; ++k) {
                    const bool live = (mask >> (PIECE_INSTRS - 1 - k)) & 1u;
                    const uint32_t b_lo = __ballot_sync(0xffffffffu, live), b_ls = b_lo & short_lanes;
                    if (live) {
                        q.lo[at[k] + __popc(b_lo & below)] = x & 0xFFFFu;
                        if (!(flag & 2u)) q.ls[as[k] + __popc(b_ls & below)] = x & 0xFFFFu;
                    }
                    at[k] += __popc(b_lo);
                    as[k] += __popc(b_ls);
                }
            }
            __syncwarp();
        }
        uint32_t my_n = 0;  // lane k: length of the short list of instruction k
#pragma unroll
        for (uint32_t k = 0; k < PIECE_INSTRS; ++k)
            if (lane == k) my_n = at[k] - my_lo - ls_mul;
        if (lane < po.ni)
            q.irec[i0 + lane] = make_uint4(my_lo - ls_sub - (i0 + lane) * ls_mul,
                                           my_n | (nd_k << 16) | (min(n_reads, 127u) << 24) | (th0 << 31), v0, o_k);
        return;
    }
    pdl_wait();
    role -= n_list;
    if (role < q.nC) {  // walk events of a chunk: entry occupancy (ascending vreg id), then instruction by instruction
        const uint32_t c = role, b = q.chunk_blk[c], p0 = q.chunk_piece_off[c];
        const size_t base = q.cev_off[c];
        const uint32_t n_entry = q.centry_cnt[c], n_ev = n_entry + q.chunk_ev[c];
        if (warp == 0)
            warp_bits(q.Wv, lane, [&](uint32_t w) { return live_before(q, c, p0, p0, w) & ~q.blk_th[(size_t)b * q.Wv + w]; },
                      [&](uint32_t rank, uint32_t v) { put_event(q, base + rank, v, q.width[v], true, true); });
        const uint32_t i1 = q.chunk_i1[c];
        for (uint32_t i = q.chunk_i0[c] + (tid + LV_NT - 32) % LV_NT; i < i1; i += LV_NT) {
            const size_t at = base + n_entry + q.ev_rel[i];
            instr_events(q, i, [&](uint32_t e, uint32_t v, bool test, bool toggle) { put_event(q, at + e, v, q.width[v], test, toggle); },
                         [&](uint32_t o) {  // listed (in any order) for the exact counts of through-set collisions
                             uint32_t s = q.chunk_short_off[c];
                             while (s + 1 < q.chunk_short_off[c + 1] && q.piece_i0[q.short_p0[s + 1]] <= i) ++s;
                             const uint32_t v = q.op_vreg[o], member = bit_get(q.blk_th + (size_t)b * q.Wv, v);
                             q.el[q.op_off[q.blk_off[b]] + atomicAdd(q.el_count + b, 1u)] = make_uint4(i, c, v | (member << 31), s);
                         });
        }
        // no-ops up to a whole group, and two no-op groups behind the last chunk (the walk reads ahead)
        const uint32_t n_pad = (8u - (n_ev & 7u)) % 8u + (c == q.nC - 1 ? 16u : 0u);
        if (tid < n_pad) put_event(q, base + n_ev + tid, q.V, 1u, false, false);
        return;
    }
    role -= q.nC;
    if (role < n_short) {
        // Events of a short chunk, 4 bytes each: vreg | width << 16 | test << 24 | toggle << 25; 32 short chunks side
        // by side, step by step, padded with zeros to the longest of the 32.  What is occupied on entry (and not
        // through the whole block) is a list of its own, vreg | short chunk << 16: those need no order.
        const uint32_t s = role * LV_WARPS + warp;
        const uint32_t steps = q.sev_off[(s >> 5) + 1] - q.sev_off[s >> 5];
        uint32_t *dst = q.sev + (size_t)q.sev_off[s >> 5] * 32 + (s & 31);
        uint32_t n = 0;
        if (s < q.nS) {
            const uint32_t p = q.short_p0[s], c = q.piece_chunk[p], b = q.chunk_blk[c], p0 = q.chunk_piece_off[c];
            const uint32_t ent0 = q.sen_off[s];
            warp_bits(q.Wv, lane, [&](uint32_t w) { return live_before(q, c, p, p0, w) & ~q.blk_th[(size_t)b * q.Wv + w]; },
                      [&](uint32_t rank, uint32_t v) { q.sen[ent0 + rank] = v | (s << 16); });
            const uint32_t i0 = q.piece_i0[p];
            const uint32_t i1 = s + 1 < q.chunk_short_off[c + 1] ? q.piece_i0[q.short_p0[s + 1]] : q.chunk_i1[c];
            const uint32_t ev0 = q.ev_rel[i0];
            for (uint32_t i = i0 + lane; i < i1; i += 32) {
                const uint32_t at = q.ev_rel[i] - ev0;
                instr_events(q, i, [&](uint32_t e, uint32_t v, bool test, bool toggle) {
                    dst[(size_t)(at + e) * 32] = v | ((uint32_t)q.width[v] << 16) | (test ? 1u << 24 : 0u) | (toggle ? 1u << 25 : 0u);
                }, [](uint32_t) {});
            }
            n = q.short_ev[s];
        }
        for (uint32_t e = n + lane; e < steps; e += 32) dst[(size_t)e * 32] = 0;
        return;
    }
    role -= n_short;
    if (role < q.nB) {  // through-set list of a block: vreg | width << 16
        const uint32_t b = role;
        if (warp == 0)
            warp_bits(q.Wv, lane, [&](uint32_t w) { return q.blk_th[(size_t)b * q.Wv + w]; },
                      [&](uint32_t rank, uint32_t v) { q.th[q.th_off[b] + rank] = v | ((uint32_t)q.width[v] << 16); });
    }
}

// --------------------------------------------------------------------------- host
namespace {
template <typename T>
cudaError_t pool_get(VlArena &arena, T **out, size_t n)
{
    return arena.alloc((void **)out, std::max<size_t>(n, 1) * sizeof(T) + 64);
}

}  // namespace
#define KEEP(out, n) VL_CUDA(p, pool_get(p->live_arena, out, n))
#define LAYOUT(out, n) VL_CUDA(p, pool_get(p->layout_arena, out, n))

#define LAUNCH(kernel, grid, nt, smem, st, ...)                 \
    do {                                                        \
        if ((grid) > 0) {                                       \
            kernel<<<(grid), (nt), (smem), (st)>>>(__VA_ARGS__); \
            g_vl_launches.fetch_add(1);                         \
        }                                                       \
    } while (0)

// About the memory of a run that does not depend on the list lengths (live_begin); small: k_small takes the program.
static size_t live_bytes(const vl_program *p, bool small)
{
    const size_t sets = small ? (size_t)p->nP + p->nC + 4 * (size_t)p->nB : 3 * (size_t)p->nP + 4 * (size_t)p->nC + 5 * (size_t)p->nB;
    return 4 * sets * p->Wv + (size_t)p->nI * 28 + (size_t)p->nO * 18 +
           (size_t)p->nC * 40 + (size_t)p->nS * 16 + (size_t)p->nB * 24 + 40 * 512;
}

// Chunks, pieces, short chunks and segments depend on the program and on the chunk size only: they are laid
// out (and uploaded, in one copy) when the chunk size changes, not on every call.
static int vl_layout(vl_program *p, cudaStream_t st)
{
    if (p->layout_chunk_instrs == p->chunk_instrs) return VL_OK;
    const uint32_t nB = p->nB;
    p->layout_chunk_instrs = 0;
    p->sizes_known = false;
    VL_CUDA(p, cudaDeviceSynchronize());  // earlier work (on any stream) may still read the old layout
    p->layout_arena.reset();
    p->tables_built = false;
    p->d_vreg16 = nullptr; p->d_first8 = nullptr; p->d_opoff = nullptr; p->d_first4 = nullptr;
    p->d_first_def_instr = nullptr; p->d_vinfo = nullptr; p->d_first_occ = nullptr;
    std::vector<uint32_t> c_i0, c_i1, c_blk, blk_c_off(nB + 1, 0), p_i0, p_o0, p_chunk, c_p_off, seg_c0, blk_seg_off(nB + 1, 0);
    for (uint32_t b = 0; b < nB; ++b) {
        const uint64_t s = p->h_blk_off[b], n = p->h_blk_off[b + 1] - s;
        uint64_t nc = (n + p->chunk_instrs - 1) / p->chunk_instrs;
        // a thread block of the walk takes 8 chunks, one per warp: a chunk count that is a multiple
        // of 8 keeps the warps equally busy (the chunks get a little shorter than asked for)
        if (nc > 4 && n >= 8 * 16) nc = (nc + 7) / 8 * 8;
        for (uint64_t j = 0; j < nc; ++j) {
            const uint32_t i0 = (uint32_t)(s + j * n / nc), i1 = (uint32_t)(s + (j + 1) * n / nc);
            c_p_off.push_back((uint32_t)p_i0.size());
            // Instructions of more operands than half a piece's would each be a piece, with three sets of all vregs: in a long
            // program they share one, whose operands are taken instruction by instruction.  (32,000 instructions of 24
            // operands each, 500 and 10,666 vregs, a run of theirs: 221 us and 1,663, so 155 and 1,087)
            auto many = [&](uint32_t i) { return p->nI > LIVE_SMALL_INSTRS && p->h_op_off[i + 1] - p->h_op_off[i] > PIECE_OPERANDS / 2; };
            for (uint32_t q0 = i0, q1; q0 < i1; q0 = q1) {
                for (q1 = q0 + 1; q1 < i1 && q1 < q0 + PIECE_INSTRS && many(q0) && many(q1);) ++q1;
                if (q1 == q0 + 1)
                    while (q1 < i1 && q1 < q0 + PIECE_INSTRS && p->h_op_off[q1 + 1] - p->h_op_off[q0] <= PIECE_OPERANDS) ++q1;
                p_i0.push_back(q0);
                p_chunk.push_back((uint32_t)c_i0.size());
            }
            c_i0.push_back(i0);
            c_i1.push_back(i1);
            c_blk.push_back(b);
        }
        blk_c_off[b + 1] = (uint32_t)c_i0.size();
    }
    c_p_off.push_back((uint32_t)p_i0.size());
    p_i0.push_back(p->nI);
    for (uint32_t i : p_i0) p_o0.push_back(p->h_op_off[i]);
    p->wide_pieces = false;
    for (size_t j = 0; j + 1 < p_o0.size(); ++j) p->wide_pieces = p->wide_pieces || p_o0[j + 1] - p_o0[j] > PIECE_OPERANDS;
    const uint32_t nC = p->nC = (uint32_t)c_i0.size();
    p->nP = (uint32_t)p_chunk.size();
    // segments of k_flow: at most about 256 of them beside one per block
    const uint32_t seg = std::max<uint32_t>(SEG_CHUNKS, (nC + 255) / 256);
    for (uint32_t b = 0; b < nB; ++b) {
        for (uint32_t c = blk_c_off[b]; c < blk_c_off[b + 1]; c += seg) seg_c0.push_back(c);
        blk_seg_off[b + 1] = (uint32_t)seg_c0.size();
    }
    p->nSeg = (uint32_t)seg_c0.size();
    seg_c0.push_back(nC);
    // short chunks: as few pieces as keep their number within SHORT_CHUNKS, equally long inside a chunk
    std::vector<uint32_t> s_p0, c_s_off(nC + 1, 0), s_blk, s_i0, b_s_off, s_chunk;
    for (uint32_t r = std::max(1u, (p->nP + SHORT_CHUNKS - 1) / SHORT_CHUNKS);; ++r) {
        uint64_t total = 0;
        for (uint32_t c = 0; c < nC; ++c) total += (c_p_off[c + 1] - c_p_off[c] + r - 1) / r;
        if (total > SHORT_CHUNKS && total > nC) continue;  // (a chunk is the longest they can get)
        for (uint32_t c = 0; c < nC; ++c) {
            const uint32_t n = c_p_off[c + 1] - c_p_off[c], k = (n + r - 1) / r;
            for (uint32_t j = 0; j < k; ++j) {
                s_p0.push_back(c_p_off[c] + (uint32_t)((uint64_t)n * j / k));
                s_blk.push_back(c_blk[c]);
                s_chunk.push_back(c);
            }
            c_s_off[c + 1] = (uint32_t)s_p0.size();
        }
        break;
    }
    p->nS = (uint32_t)s_p0.size();
    for (uint32_t x : s_p0) s_i0.push_back(p_i0[x]);
    s_i0.push_back(p->nI);
    for (uint32_t b = 0; b <= nB; ++b) b_s_off.push_back(c_s_off[blk_c_off[b]]);
    p->short_len = 1;
    for (uint32_t j = 0; j < p->nS; ++j) p->short_len = std::max(p->short_len, s_i0[j + 1] - s_i0[j]);
    // shares of the thread blocks of k_small: whole chunks, about equally many pieces; then that of a single one
    std::vector<uint32_t> share, share_c0(SMALL_BLOCKS + 1, nC);
    p->share_pieces = p->share_ops = 0;
    for (uint32_t r = 0; r < SMALL_BLOCKS; ++r) {
        const uint32_t want = (uint32_t)((uint64_t)p->nP * r / SMALL_BLOCKS);
        share_c0[r] = (uint32_t)(std::lower_bound(c_p_off.begin(), c_p_off.end(), want) - c_p_off.begin());
    }
    share_c0.push_back(0);
    share_c0.push_back(nC);
    for (uint32_t c : share_c0)
        for (uint32_t x : {c, c_p_off[c], p_i0[c_p_off[c]], p_o0[c_p_off[c]]}) share.push_back(x);
    for (uint32_t r = 0; r < SMALL_BLOCKS; ++r) {
        p->share_pieces = std::max(p->share_pieces, share[4 * r + 5] - share[4 * r + 1]);
        p->share_ops = std::max(p->share_ops, share[4 * r + 7] - share[4 * r + 3]);
    }
    std::vector<uint32_t> all;
    struct Part { uint32_t **dst; const std::vector<uint32_t> *v; };
    uint32_t *d_share = nullptr, *none = nullptr;
    const Part parts[] = {{&d_share, &share},
                          // (side by side, see SmallSmem)
                          {&p->d_blk_chunk_off, &blk_c_off}, {&p->d_chunk_piece_off, &c_p_off}, {&p->d_chunk_blk, &c_blk},
                          {&p->d_chunk_short_off, &c_s_off}, {&p->d_short_p0, &s_p0}, {&p->d_short_chunk, &s_chunk}, {&none, &p->h_blk_off},
                          {&none, &p->h_succ_off}, {&none, &p->h_succ},
                          {&p->d_chunk_i0, &c_i0}, {&p->d_chunk_i1, &c_i1}, {&p->d_piece_i0, &p_i0}, {&p->d_piece_o0, &p_o0},
                          {&p->d_piece_chunk, &p_chunk}, {&p->d_seg_c0, &seg_c0}, {&p->d_blk_seg_off, &blk_seg_off}, {&p->d_short_blk, &s_blk},
                          {&p->d_short_i0, &s_i0}, {&p->d_blk_short_off, &b_s_off}};
    for (const Part &x : parts) {
        all.insert(all.end(), x.v->begin(), x.v->end());
        all.resize((all.size() + 4) & ~(size_t)3);  // (at least one word behind every array)
    }
    uint32_t *dev = nullptr;
    // The operand words lie beside the tables; those of a long program in the slab of the runs' memory: they would take a program
    // of 32,000 instructions one device allocation more, 300 us of the first run's 1,200.  (There for every program: a run of a
    // short one, its memory untouched for a while, 1 % slower.)
    const bool beside = p->nO <= 65536;
    p->layout_arena.hint = all.size() * 4 + (size_t)p->V * 12 + (beside ? (size_t)p->nO * 4 : 0) + (size_t)p->nOp8 * 3 + (size_t)p->nOpT * 5 + 16384;
    LAYOUT(&dev, all.size());
    VL_CUDA(p, cudaMemcpy(dev, all.data(), all.size() * 4, cudaMemcpyHostToDevice));
    size_t at = 0;
    for (const Part &x : parts) {
        *x.dst = dev + at;
        at = (at + x.v->size() + 4) & ~(size_t)3;
    }
    p->d_share = reinterpret_cast<uint4 *>(d_share);
    vl_free_liveness(p);
    p->live_arena.clear();
    if (beside) {
        LAYOUT(&p->d_op_word, (size_t)p->nO);
    } else {
        p->live_arena.hint = live_bytes(p, false) + (size_t)p->nO * 4 + 512;
        KEEP(&p->d_op_word, (size_t)p->nO);
    }
    p->live_arena.keep();
    LAUNCH(k_operand_words, (p->nP + NT / 32 - 1) / (NT / 32), NT, 0, st, p->nP, p->d_piece_i0, p->d_op_off, p->d_ndefs, p->d_op_vreg, p->d_op_word);
    VL_CUDA(p, cudaGetLastError());
    p->words_new = true;
    const uint32_t Wp = (p->P + p->wmax + 31) / 32 + 1;
    p->use_th = (nB <= 32 && (uint64_t)nB * VL_MAX_GROUP * Wp * 4 <= 24 * 1024) ? 1 : 0;
    p->layout_chunk_instrs = p->chunk_instrs;
    return VL_OK;
}

// What a run's launches need besides the arguments.
struct LiveShape {
    bool wide = false, small = false;  // small: k_small takes the program
    size_t small_smem = 0;
    uint32_t set_warps = PC_WARPS, sets = 0, flows = 0, counts = 0, offs = 0, fills = 0;
    size_t sets_smem = 0, flow_smem = 0, count_smem = 0, fill_smem = 0;
    void add(const LiveShape &o)
    {
        wide = wide || o.wide;
        small_smem = std::max(small_smem, o.small_smem);
        set_warps = std::min(set_warps, o.set_warps);
        sets = std::max(sets, o.sets); flows = std::max(flows, o.flows); counts = std::max(counts, o.counts);
        offs = std::max(offs, o.offs); fills = std::max(fills, o.fills);
        sets_smem = std::max(sets_smem, o.sets_smem); flow_smem = std::max(flow_smem, o.flow_smem);
        count_smem = std::max(count_smem, o.count_smem);
        fill_smem = std::max(fill_smem, o.fill_smem);
    }
};

// The memory of a run that does not depend on the list lengths, and its arguments.
static int live_begin(vl_program *p, LiveArgs &q, LiveShape &sh, cudaStream_t st)
{
    vl_free_liveness(p);
    const uint32_t nB = p->nB, nI = p->nI, V = p->V, nO = p->nO, Wv = p->Wv, nC = p->nC, nP = p->nP;

    q = LiveArgs{};
    sh.small_smem = q.small.init(nB, p->nE, nC, p->nS, Wv, p->share_pieces, p->share_ops);
    sh.small = nI <= LIVE_SMALL_INSTRS && nC && sh.small_smem <= SMALL_SMEM;
    p->live_arena.hint = live_bytes(p, sh.small);  // what follows, in one slab
    // ---- results and tables that do not depend on the list lengths
    KEEP(&p->d_blk_in, (size_t)2 * nB * Wv);  // live-in rows, then live-out rows
    p->d_blk_out = p->d_blk_in + (size_t)nB * Wv;
    KEEP(&p->d_lo_off, (size_t)nI + 1);
    KEEP(&p->d_opflags, (size_t)nO);
    // the operand tables of the verify kernels depend on the program alone: made by the first run, kept
    if (!p->d_opoff) {
        LAYOUT(&p->d_first_def_instr, (size_t)V);
        LAYOUT(&p->d_first_occ, (size_t)V);
        LAYOUT(&p->d_vreg16, (size_t)p->nOp8 + 8);
        LAYOUT(&p->d_first8, (size_t)p->nOp8 / 8);
        LAYOUT(&p->d_first4, (size_t)p->nOpT / 4);
        LAYOUT(&p->d_vinfo, (size_t)V);
        LAYOUT(&p->d_opoff, (size_t)p->nOpT / 4);
    }
    KEEP(&p->d_cev_off, (size_t)nC + 1);
    KEEP(&p->d_th_off, (size_t)nB + 1);
    KEEP(&p->d_th_cnt, (size_t)nB);
    KEEP(&p->d_ls_adj, (size_t)nB);
    KEEP(&p->d_blk_th, (size_t)nB * Wv);
    KEEP(&p->d_el, (size_t)nO);  // at most one entry per definition
    KEEP(&p->d_el_count, (size_t)nB);
    KEEP(&p->d_sev_off, (size_t)(p->nS + 31) / 32 + 1);
    KEEP(&p->d_sen_off, (size_t)p->nS + 1);
    KEEP(&p->d_irec, (size_t)nI);

    q.nB = nB; q.nI = nI; q.V = V; q.nE = p->nE; q.Wv = Wv; q.nC = nC; q.nP = nP; q.nS = p->nS; q.nSeg = p->nSeg;
    q.use_th = p->use_th;
    q.op_off = p->d_op_off; q.op_vreg = p->d_op_vreg; q.succ_off = p->d_succ_off; q.succ = p->d_succ; q.blk_off = p->d_blk_off;
    q.ndefs = p->d_ndefs; q.width = p->d_width;
    q.chunk_i0 = p->d_chunk_i0; q.chunk_i1 = p->d_chunk_i1; q.chunk_blk = p->d_chunk_blk; q.blk_chunk_off = p->d_blk_chunk_off;
    q.piece_i0 = p->d_piece_i0; q.piece_o0 = p->d_piece_o0; q.op_word = p->d_op_word; q.piece_chunk = p->d_piece_chunk; q.chunk_piece_off = p->d_chunk_piece_off;
    q.seg_c0 = p->d_seg_c0; q.blk_seg_off = p->d_blk_seg_off; q.short_p0 = p->d_short_p0; q.chunk_short_off = p->d_chunk_short_off;
    if (!sh.small) {  // (k_small keeps these in shared memory)
        KEEP(&q.piece_use, (size_t)nP * Wv);
        KEEP(&q.piece_def, (size_t)nP * Wv);
        KEEP(&q.chunk_use, (size_t)nC * Wv);
        KEEP(&q.chunk_def, (size_t)nC * Wv);
        KEEP(&q.chunk_end, (size_t)nC * Wv);
        KEEP(&q.blk_touch, (size_t)nB * Wv);
        KEEP(&q.chunk_lo, (size_t)nC);
        KEEP(&q.short_ent, (size_t)p->nS);
        KEEP(&q.counters, 1);
    }
    KEEP(&q.piece_end, (size_t)nP * Wv);
    KEEP(&q.chunk_entry, (size_t)nC * Wv);
    KEEP(&q.lo_rel, (size_t)nI);
    KEEP(&q.ev_rel, (size_t)nI);
    KEEP(&q.chunk_ev, (size_t)nC);
    KEEP(&q.chunk_lo0, (size_t)nC + 1);
    KEEP(&q.centry_cnt, (size_t)nC);
    KEEP(&q.short_ev, (size_t)p->nS);
    const uint32_t fgrid = (Wv + 31) / 32;
    size_t flow_smem = (((size_t)4 * nB + 2 * (size_t)p->nSeg) * 32 + nB + 1 + p->nE) * 4;
    if (flow_smem > 200 * 1024 && !sh.small) {
        KEEP(&q.flow_scratch, flow_smem / 4 * fgrid);
        flow_smem = 0;
    }
    if (!p->tables_built) {
        VL_CUDA(p, cudaMemsetAsync(p->d_first_occ, 0xFF, std::max<size_t>(V, 1) * 4, st));
        VL_CUDA(p, cudaMemsetAsync(p->d_first_def_instr, 0xFF, std::max<size_t>(V, 1) * 4, st));
    }
    q.blk_in = p->d_blk_in; q.blk_out = p->d_blk_out; q.lo_off = p->d_lo_off; q.opflags = p->d_opflags;
    q.cev_off = p->d_cev_off; q.th_off = p->d_th_off; q.th_cnt = p->d_th_cnt; q.ls_adj = p->d_ls_adj; q.blk_th = p->d_blk_th;
    q.el = p->d_el; q.el_count = p->d_el_count; q.status = p->d_status; q.sev_off = p->d_sev_off; q.sen_off = p->d_sen_off; q.irec = p->d_irec;
    q.host_out = p->h_live;
    // a bitset pair per warp of k_sets: fewer warps for programs of very many vregs
    sh.set_warps = (uint32_t)std::max<size_t>(1, std::min<size_t>(PC_WARPS, (size_t)224 * 1024 / ((size_t)2 * Wv * 4)));
    sh.sets = std::max(1u, nC); sh.flows = fgrid; sh.counts = nC; sh.offs = nC + nB;
    sh.fills = (nP + LV_WARPS - 1) / LV_WARPS + nC + ((p->nS + 31) & ~31u) / LV_WARPS + nB;
    sh.sets_smem = (size_t)sh.set_warps * 2 * Wv * 4;
    sh.wide = p->wide_pieces;
    sh.count_smem = p->wide_pieces ? (size_t)PC_WARPS * 2 * Wv * 4 : 0;
    q.wide_smem = sh.count_smem <= 40 * 1024;
    if (!q.wide_smem) sh.count_smem = 0;
    sh.flow_smem = flow_smem;
    q.share = p->d_share; q.small_tab = p->d_blk_chunk_off;
    sh.fill_smem = (size_t)LV_WARPS * (2 * Wv + FILL_WARP_WORDS) * 4;
    return VL_OK;
}

// The list lengths: read on the first run with this layout (its first four kernels have finished); later runs
// allocate from the lengths they remember (same program, same layout) and only compare at the end.
static int live_lengths(vl_program *p, LiveArgs &q)
{
    if (!p->sizes_known) {
        const uint32_t status = p->h_live[0];
        unsigned long long tot[LV_TOTALS];
        memcpy(tot, p->h_live + 2, sizeof(tot));
        if (status & ST_NO_CONVERGE) return VL_ERR_NO_CONVERGE;
        if (status & ST_NOT_STRICT) return VL_ERR_NOT_STRICT;
        if (status & ST_SIZE_OVERFLOW) return VL_ERR_UNSUPPORTED;
        if (tot[LV_TOT_EV] > 0xFFFFFFF0ull || tot[LV_TOT_SEV] > 0xFFFFFFF0ull || tot[LV_TOT_SEN] > 0xFFFFFFF0ull)
            return VL_ERR_UNSUPPORTED;
        memcpy(p->known, tot, sizeof(tot));
    }
    p->lo_len = p->known[LV_TOT_LO];
    p->live_arena.hint = 4 * (p->known[LV_TOT_LO] + p->known[LV_TOT_LS] + p->known[LV_TOT_TH] + p->known[LV_TOT_SEV] + p->known[LV_TOT_SEN]) +
                         18 * p->known[LV_TOT_EV] + 9 * 512;
    KEEP(&p->d_lo, (size_t)p->lo_len);
    KEEP(&p->d_ls, (size_t)p->known[LV_TOT_LS]);
    KEEP(&p->d_ev, (size_t)(p->known[LV_TOT_EV] / 8 + 2) * 7);  // two no-op groups behind the last chunk
    if (vl_eight_takes(p)) KEEP(&p->d_ev8, (size_t)p->known[LV_TOT_EV] + 16);
    KEEP(&p->d_th, (size_t)p->known[LV_TOT_TH]);
    KEEP(&p->d_sev, (size_t)p->known[LV_TOT_SEV]);
    KEEP(&p->d_sen, (size_t)p->known[LV_TOT_SEN]);
    q.lo = p->d_lo; q.ls = p->d_ls; q.ev = p->d_ev; q.ev8 = p->d_ev8; q.th = p->d_th; q.sev = p->d_sev; q.sen = p->d_sen;
    return VL_OK;
}

// The operand tables of the verify kernels (first run).
static int live_tables(vl_program *p, cudaStream_t st)
{
    p->bank_fast = ((p->B == 1 || p->B == 2 || p->B == 4) && !p->bank_many) ? 1 : 0;
    if (p->tables_built) return VL_OK;
    const uint32_t nI = p->nI, V = p->V;
    LAUNCH(k_first_occ, (nI + NT - 1) / NT, NT, 0, st, nI, p->d_op_off, p->d_ndefs, p->d_op_vreg, p->d_first_occ,
           p->d_first_def_instr);
    LAUNCH(k_vreg_info, (V + NT - 1) / NT, NT, 0, st, V, p->d_width, p->d_first_occ, p->d_first_def_instr, p->d_vinfo);
    LAUNCH(k_operand_tables, (p->nOpT / 8 + NT - 1) / NT, NT, 0, st, p->nO, p->nOp8, p->nOpT / 8, V, p->d_op_vreg, p->d_first_occ,
           p->d_vreg16, p->d_first8, p->d_opoff, p->d_first4);
    VL_CUDA(p, cudaGetLastError());
    p->tables_built = true;
    return VL_OK;
}

// k_small for the runs of n <= N programs, C thread blocks each.
template <int N, int C>
static int launch_small(vl_program *p, const LiveMany<N> &many, uint32_t n, size_t smem, cudaStream_t st, bool overlap)
{
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = C; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(C, n); cfg.blockDim = SMALL_NT; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = at; cfg.numAttrs = C > 1 ? 2 : 1;
    VL_CUDA(p, (allow_smem<k_small<N, C>, SMALL_SMEM>(p->device)));
    g_vl_launches.fetch_add(1);
    VL_CUDA(p, cudaLaunchKernelEx(&cfg, k_small<N, C>, many));
    return VL_OK;
}

// The kernels of the runs of n <= N programs up to the list lengths, or the last one.
template <int N>
static int live_launch(vl_program *const *progs, uint32_t n, const LiveArgs *args, const LiveShape *shapes, bool fill,
                       cudaStream_t st)
{
    vl_program *p = progs[0];
    LiveMany<N> many;
    if (fill) {
        LiveShape sh;
        for (uint32_t j = 0; j < n; ++j) {
            sh.add(shapes[j]);
            many.p[j] = args[j];
        }
        VL_CUDA(p, (allow_smem<k_fill<N>, 227 * 1024>(p->device)));
        VL_CUDA(p, launch_overlap(k_fill<N>, dim3(sh.fills, n), LV_NT, sh.fill_smem, st, true, many));
        return VL_OK;
    }
    for (const bool small : {true, false}) {
        LiveShape sh;
        uint32_t m = 0;
        // The first kernel of a run reads the operand words before it waits for the stream: behind the kernel that makes them it
        // starts when that one has ended.  (A wait of the host in between: 82.3 us for the first run of 64 instructions, 79.4
        // without operand words.)
        bool overlap = true;
        for (uint32_t j = 0; j < n; ++j) {
            if (shapes[j].small != small) continue;
            overlap = overlap && !progs[j]->words_new;
            sh.add(shapes[j]);
            many.p[m++] = args[j];
        }
        if (!m) continue;
        if (small) {
            SmallSmem one;
            const uint32_t one_smem = one.init(p->nB, p->nE, p->nC, p->nS, p->Wv, p->nP, p->nO);
            int rc;
            if (N == 1 && p->nP <= SMALL_ONE_PIECES && one_smem <= SMALL_SMEM) {
                many.p[0].small = one;
                rc = launch_small<N, N == 1 ? 1 : SMALL_BLOCKS>(p, many, m, one_smem, st, overlap);
            } else {
                rc = launch_small<N, SMALL_BLOCKS>(p, many, m, sh.small_smem, st, overlap);
            }
            if (rc != VL_OK) return rc;
            continue;
        }
        VL_CUDA(p, (allow_smem<k_sets<N>, 227 * 1024>(p->device)));
        VL_CUDA(p, launch_overlap(k_sets<N>, dim3(sh.sets, m), sh.set_warps * 32, sh.sets_smem, st, overlap, many));
        VL_CUDA(p, (allow_smem<k_flow<N>, 227 * 1024>(p->device)));
        VL_CUDA(p, launch_overlap(k_flow<N>, dim3(sh.flows, m), FLOW_WARPS * 32, sh.flow_smem, st, true, many));
        if (sh.counts && sh.wide) VL_CUDA(p, launch_overlap(k_count<N, true>, dim3(sh.counts, m), PC_NT, sh.count_smem, st, true, many));
        else if (sh.counts) VL_CUDA(p, launch_overlap(k_count<N, false>, dim3(sh.counts, m), PC_NT, 0, st, true, many));
        VL_CUDA(p, launch_overlap(k_offsets<N>, dim3(sh.offs, m), OFF_NT, 0, st, true, many));
    }
    return VL_OK;
}

// The runs of n programs, LV_MANY of them per launch, the launches spread over the n_streams streams.  Everything is
// recomputed on the device every time.  One event is recorded per stream; the programs that run on it share it (64
// programs of one call: 2 events instead of 64).  The first program with an error ends the call: those behind it keep what
// an earlier run left them (their results are computed once more, the same), or stay without a run.
int vl_liveness_impl(vl_program *const *progs, uint32_t n, const cudaStream_t *streams, uint32_t n_streams)
{
    std::vector<LiveArgs> args(n);
    std::vector<LiveShape> shapes(n);
    std::vector<uint8_t> had_run(n);
    bool lengths_known = true;
    int rc = VL_OK, err = VL_OK;
    const uint32_t per = n == 1 ? 1 : LV_MANY;
    auto stream_of = [&](uint32_t j) { return (j / per) % n_streams; };
    for (uint32_t j = 0; j < n; ++j) {
        vl_program *p = progs[j];
        vl_live_settle(p);  // the pinned words of an earlier run are about to be reused
        had_run[j] = p->live_ok;
        err = vl_layout(p, streams[stream_of(j)]);
        if (err == VL_OK && !p->h_live && !(p->h_live = (uint32_t *)vl_pinned_get())) err = VL_ERR_CUDA;
        if (err == VL_OK) err = live_begin(p, args[j], shapes[j], streams[stream_of(j)]);
        if (err != VL_OK) {
            // (its next run may be on another stream than the kernel that makes its operand words)
            if (p->words_new) cudaStreamSynchronize(streams[stream_of(j)]);
            p->words_new = false;
            n = j;  // (those behind it are untouched)
            break;
        }
        lengths_known = lengths_known && p->sizes_known;
    }
    auto launch = [&](bool fill) -> int {
        for (uint32_t j = 0; j < n; j += per) {
            const cudaStream_t st = streams[stream_of(j)];
            const uint32_t m = std::min(per, n - j);
            const int r = m == 1 ? live_launch<1>(progs + j, 1, &args[j], &shapes[j], fill, st)
                                 : live_launch<LV_MANY>(progs + j, m, &args[j], &shapes[j], fill, st);
            if (r != VL_OK) return r;
        }
        return VL_OK;
    };
    rc = launch(false);
    for (uint32_t j = 0; j < n; ++j) {
        if (rc != VL_OK && progs[j]->words_new) cudaStreamSynchronize(streams[stream_of(j)]);
        progs[j]->words_new = false;
    }
    if (rc != VL_OK) return rc;
    if (!lengths_known)
        for (uint32_t s = 0; s < n_streams; ++s) VL_CUDA(progs[0], cudaStreamSynchronize(streams[s]));
    std::vector<vl_program *> run;  // the programs that the last kernel is launched for
    for (uint32_t j = 0; j < n; ++j) {
        if (err != VL_OK && !had_run[j]) continue;
        const int r = live_lengths(progs[j], args[j]);
        if (r != VL_OK) {
            if (err == VL_OK) err = r;
            continue;
        }
        args[run.size()] = args[j];
        shapes[run.size()] = shapes[j];
        run.push_back(progs[j]);
    }
    if (run.size() < n && lengths_known)  // (a program may move to another stream)
        for (uint32_t s = 0; s < n_streams; ++s) VL_CUDA(progs[0], cudaStreamSynchronize(streams[s]));
    progs = run.data();
    n = (uint32_t)run.size();
    if ((rc = launch(true)) != VL_OK) return rc;
    for (uint32_t j = 0; j < n; ++j)
        if ((rc = live_tables(progs[j], streams[stream_of(j)])) != VL_OK) return rc;
    for (uint32_t j = 0; j < n; ++j) {
        vl_program *p = progs[j];
        if (j % per == 0 && j / per < n_streams) {  // the first program of a stream
            if (!p->ev_live || p->ev_live.use_count() > 1) {
                auto e = std::make_shared<VlEvent>();
                VL_CUDA(p, cudaEventCreateWithFlags(&e->ev, cudaEventDisableTiming));
                p->ev_live = e;
            }
            VL_CUDA(p, cudaEventRecord(p->ev_live->ev, streams[stream_of(j)]));
        }
        p->live_done = progs[stream_of(j) * per]->ev_live;
        p->live_pending = true;
        p->live_ok = true;
    }
    if (n) VL_CUDA(progs[0], cudaGetLastError());
    if (lengths_known) return err;  // lengths remembered from an earlier run: checked when the results are used
    for (uint32_t j = 0; j < n; ++j) {
        if ((rc = vl_live_settle(progs[j])) != VL_OK) return rc;
        progs[j]->sizes_known = true;
    }
    return err;
}

int vl_live_settle(vl_program *p)
{
    if (!p->live_pending) return VL_OK;
    p->live_pending = false;
    p->live_ok = false;
    const std::shared_ptr<VlEvent> done = std::move(p->live_done);
    VL_CUDA(p, cudaEventSynchronize(done->ev));
    const uint32_t status = p->h_live[0];
    unsigned long long tot[LV_TOTALS];
    memcpy(tot, p->h_live + 2, sizeof(tot));
    if (status & ST_NO_CONVERGE) return VL_ERR_NO_CONVERGE;
    if (status & ST_NOT_STRICT) return VL_ERR_NOT_STRICT;
    if (status & ST_SIZE_OVERFLOW) return VL_ERR_UNSUPPORTED;
    if (memcmp(tot, p->known, sizeof(tot)) != 0) {
        // the lengths the run allocated from do not fit what it computed: the next run measures again
        p->sizes_known = false;
        return VL_ERR_CUDA;
    }
    p->live_ok = true;
    return VL_OK;
}
