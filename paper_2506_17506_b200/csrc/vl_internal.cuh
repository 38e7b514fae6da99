// Internal declarations shared by the translation units of libverilocc.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <memory>
#include <vector>

#include "verilocc.h"

// ---- per-operand flag byte written by the liveness walk (device array opflags[n_operands])
enum : uint8_t {
    OPF_DEF = 1,    // operand is a definition
    OPF_KILL = 2,   // read: the value dies here (first read of the vreg in the instruction)
    OPF_DUP = 4,    // read: same vreg read earlier by this instruction
    OPF_ELIDE = 8,  // definition of a vreg the instruction also reads and that stays live:
                    //   occupancy unchanged, no walk event
    OPF_SET = 16,   // definition: becomes occupied (live after, or several defs in the instruction)
    OPF_POST = 32,  // definition: dead, released again after the instruction's definitions
    OPF_DEAD = 64   // definition: vreg not live after the instruction
};

// ---- a walk event of k_eight: byte offset of the vreg's 16-byte table entry (bits 4 to 17), whether it tests, whether it leaves
// the occupancy as it is, and the mask of its width, at most 8 registers (0: no event)
#define EV8_OFFSET 0x3FFF0u
#define EV8_TEST 1u
#define EV8_HOLD 2u
#define EV8_MASK_SHIFT 24

enum : uint32_t { VINFO_OCCURS = 1u << 8, VINFO_DEFINED = 1u << 9 };

// ---- device status word bits (prog->d_status[0] liveness, d_status[1] verify)
enum : uint32_t {
    ST_NO_CONVERGE = 1u,
    ST_NOT_STRICT = 2u,
    ST_MANY_USES = 4u,      // some instruction reads more than 4 operands (bank tally takes the general path)
    ST_SIZE_OVERFLOW = 8u,  // a list length does not fit 32 bits
    ST_DEVICE_WAIT = 16u    // a bounded wait in a verify kernel ran out
};

#define VL_MAX_GROUP 8
#define VL_KNOWN_LS 3   // vl_program::known: short-list entries
#define VL_KNOWN_SEN 5  // and entries of the short chunks
#define VL_LANES 8  // internal streams that the passes of device-resident verify calls can be spread over
#define VL_LIVE_STREAM VL_LANES      // index of the internal stream a single vl_liveness call runs on
#define VL_STREAMS (VL_LANES + 1)    // the lanes, the liveness stream

// Device memory pool of a program handle: slabs are kept across calls, so that a repeated
// vl_liveness on the same handle allocates nothing.
struct VlArena {
    struct Slab { char *ptr; size_t size; };
    std::vector<Slab> slabs;
    size_t cur = 0, off = 0;
    size_t kept_cur = 0, kept_off = 0;  // what lies in front of this place outlives reset()
    size_t hint = 0;  // what the next slab should hold (a slab costs 20 us up to 64 KB, 330 us from 1 MB on, however large)
    cudaError_t alloc(void **out, size_t bytes)
    {
        bytes = (bytes + 64 + 255) & ~(size_t)255;
        for (; cur < slabs.size(); ++cur, off = 0)
            if (off + bytes <= slabs[cur].size) {
                *out = slabs[cur].ptr + off;
                off += bytes;
                return cudaSuccess;
            }
        Slab s{nullptr, bytes > hint ? bytes : hint};
        hint = (size_t)64 << 10;
        cudaError_t e = cudaMalloc((void **)&s.ptr, s.size);
        if (e != cudaSuccess) return e;
        slabs.push_back(s);
        cur = slabs.size() - 1;
        *out = s.ptr;
        off = bytes;
        return cudaSuccess;
    }
    void keep() { kept_cur = cur; kept_off = off; }
    void reset() { cur = kept_cur; off = kept_off; }
    void clear() { kept_cur = kept_off = 0; reset(); }
    void release()
    {
        for (auto &s : slabs) cudaFree(s.ptr);
        slabs.clear();
        clear();
    }
};

// An event that several handles may wait for: the programs of a liveness batch that run on one stream share one.
struct VlEvent {
    cudaEvent_t ev = nullptr;
    ~VlEvent() { if (ev) cudaEventDestroy(ev); }
};

struct vl_program {
    int device = 0;
    uint32_t nB = 0, nI = 0, V = 0, nO = 0, nE = 0, P = 0, B = 0;
    uint32_t Wv = 0;    // 32-bit words per vreg bitset
    uint32_t nOp8 = 0;  // n_operands rounded up to 8 (at least 8)
    uint32_t nOpT = 0;  // n_operands rounded up to 4096 (whole tiles of the eight-candidate table kernel), plus 4096
    uint32_t wmax = 1;  // widest vreg
    uint32_t chunk_instrs = 160;
    uint32_t group_opt = 0;

    // chunks: every chunk lies inside one block; pieces: every piece lies inside one chunk; short chunks: runs of
    // pieces of one chunk; segments: runs of chunks of one block
    uint32_t nC = 0, nP = 0, nS = 0, nSeg = 0;
    uint32_t short_len = 1;  // instructions of the longest short chunk
    uint32_t share_pieces = 0, share_ops = 0;  // pieces and operands of the largest share of a thread block of k_small
    bool wide_pieces = false;  // some piece is an instruction of many operands (PIECE_OPERANDS, vl_liveness.cu)
    bool words_new = false;  // the kernel that makes the operand words has been launched since the last run
    uint32_t layout_chunk_instrs = 0;  // chunk size the device copies of the layout were made for (0: none)
    std::vector<uint32_t> h_blk_off, h_op_off, h_succ_off, h_succ;
    // list lengths of the last liveness run with this layout: the next run allocates from them
    bool sizes_known = false;
    unsigned long long known[6] = {0, 0, 0, 0, 0, 0};  // list entries, walk events, through-set entries, short-list entries, short-chunk events and entries

    // device copies of the program: one allocation
    void *d_blob = nullptr;
    uint32_t *d_blk_off = nullptr, *d_succ_off = nullptr, *d_succ = nullptr, *d_op_off = nullptr, *d_op_vreg = nullptr;
    uint8_t *d_ndefs = nullptr, *d_width = nullptr;
    uint32_t *d_chunk_i0 = nullptr, *d_chunk_i1 = nullptr, *d_chunk_blk = nullptr, *d_blk_chunk_off = nullptr;
    uint32_t *d_piece_i0 = nullptr, *d_piece_o0 = nullptr, *d_op_word = nullptr, *d_piece_chunk = nullptr, *d_chunk_piece_off = nullptr;
    uint32_t *d_seg_c0 = nullptr, *d_blk_seg_off = nullptr, *d_short_p0 = nullptr, *d_chunk_short_off = nullptr, *d_short_blk = nullptr, *d_short_i0 = nullptr, *d_blk_short_off = nullptr, *d_short_chunk = nullptr;
    uint4 *d_share = nullptr;

    // liveness results
    uint32_t *d_blk_in = nullptr, *d_blk_out = nullptr, *d_lo_off = nullptr, *d_lo = nullptr;
    uint64_t lo_len = 0;

    // tables consumed by the verify kernels
    uint16_t *d_vreg16 = nullptr;           // [nOp8 + 8] vreg id per operand (padding operands: id V)
    uint8_t *d_first8 = nullptr;            // [nOp8 / 8] per 8 operands: first-occurrence bits
    // the same tables for rows in dictionary form (one column per (block, vreg of the block)); made once,
    // when the handle is created
    uint32_t nD = 0, nD8 = 0, nDT = 0;  // entries; rounded up to 8 (at least 8); to whole tiles plus one
    std::vector<uint32_t> h_dict_off, h_dict_vreg;
    uint16_t *d_dict_vreg16 = nullptr;
    uint8_t *d_dict_first8 = nullptr;
    uint4 *d_dict_opoff = nullptr;
    uint8_t *d_dict_first4 = nullptr;
    uint32_t *d_dict_first_occ = nullptr; // [V] first entry of the vreg, 0xFFFFFFFF if none
    uint32_t *d_dict_instr = nullptr;     // [nD8] first instruction of the entry's block that touches its vreg
    uint4 *d_opoff = nullptr;               // [nOpT / 4] per 4 operands: byte offsets of their vregs' 16-byte table entries
    uint8_t *d_first4 = nullptr;            // [nOpT / 4] per 4 operands: first-occurrence bits
    uint8_t *d_opflags = nullptr;           // [nO]
    uint32_t *d_first_occ = nullptr;        // [V] first operand that names v, 0xFFFFFFFF if none
    uint32_t *d_first_def_instr = nullptr;  // [V] lowest instruction defining v, 0xFFFFFFFF if none
    uint32_t *d_vinfo = nullptr;            // [V] width | VINFO_OCCURS | VINFO_DEFINED
    // optional hardware rules of the Realizability check (vl_program_set_constraints)
    uint4 *d_vcons = nullptr;               // [V] (class first | class end << 16, alignment, ceil(2^32 / alignment), 0); null = no rules
    uint16_t *d_rs_prefix = nullptr;        // [P+1] reserved registers below r; null = none reserved
    uint32_t *d_th_off = nullptr, *d_th = nullptr;  // per block: vregs occupied through the whole block
    // live-after lists without the block's through-set, for the exact counts: the list of instruction i of
    // block b is ls[lo_off[i] - ls_adj[b] - i * th_cnt[b] ...), |live-after| - th_cnt[b] entries
    // per instruction, for the exact counts: {first entry of its short list, entries | definitions << 16 | reads (at most
    // 127) << 24 | first defined vreg is in the block's through-set << 31, first defined vreg, first operand}
    uint4 *d_irec = nullptr;
    uint32_t *d_ls = nullptr, *d_ls_adj = nullptr, *d_th_cnt = nullptr, *d_blk_th = nullptr;
    // definitions without a walk event: {instruction, chunk, vreg | in the block's through-set << 31, short chunk};
    // those of block b start at the index of its first operand, in any order, el_count[b] of them
    uint4 *d_el = nullptr;
    uint32_t *d_el_count = nullptr;
    uint32_t *d_cev_off = nullptr;  // [nC+1] first walk event of each chunk (every chunk padded to 8 events)
    uint32_t *d_ev8 = nullptr;      // walk events of k_eight, at the same places; null if it does not take the program
    uint4 *d_ev = nullptr;          // walk events, 112 bytes per group of 8, chunk after chunk
    // events of the short chunks, 4 bytes each, 32 short chunks side by side: steps [sev_off[g], sev_off[g + 1]) of
    // group g, [step][32]; and what is occupied when short chunk s begins, vreg | s << 16, [sen_off[s], sen_off[s + 1])
    uint32_t *d_sev_off = nullptr, *d_sev = nullptr, *d_sen_off = nullptr, *d_sen = nullptr;
    int bank_fast = 0;  // B in {1,2,4} and every instruction reads <= 4 distinct vregs
    int bank_many = 0;  // some instruction reads more than 4 distinct vregs
    uint2 *d_bank_list = nullptr;   // instructions with 2, 3, 4 distinct sources: their vreg ids, 16 bits each
    uint32_t bank_seg[4] = {0, 0, 0, 0};
    uint32_t threads_opt = 0;
    uint32_t prefetch_tiles = 3;
    uint32_t stagger_us = 12;     // start offset between the classes of the first wave of the table kernel (0 = none)
    int sm_count = 0;             // multiprocessors of the device (asked once)  // tiles the eight-candidate table kernel asks into L2 ahead of its copy ring
    uint32_t test_wait = 0;  // test hook of the table kernel's bounded wait (VL_OPT_TEST_WAIT)
    int use_th = 0;

    VlArena live_arena;             // liveness results, tables and working sets
    VlArena layout_arena;           // chunks, pieces, walk items
    uint32_t *d_status = nullptr;  // [16] device status words
    int last_cuda_error = 0;
    bool live_ok = false;
    // A repeated liveness run (same layout, lengths remembered) does not wait for the GPU: its kernels write
    // the status word and the list lengths to pinned host memory, and the next call that needs the results on
    // the host side (vl_live_settle) waits for the run and checks them.
    uint32_t *h_live = nullptr;      // pinned: [0] status, [2..13] six 64-bit totals, written by the run's kernels
    std::shared_ptr<VlEvent> ev_live;    // made by this handle, used again when no other handle waits for it
    std::shared_ptr<VlEvent> live_done;  // behind the run in flight: ev_live of this handle, or of another one of its batch
    bool live_pending = false;
    // The id of the stream that the run in flight is ordered on (ids are never used again; a caller's handle is, once its
    // stream is destroyed, and the handle of the per-thread default stream names one in every thread): the caller's, or (a long program's vl_liveness) an internal one,
    // behind what the caller's stream held when it was called.  Calls on other streams that read the results make theirs
    // wait for live_done (vl_live_join); the table kernel, which reads the program's operand tables only, runs beside the
    // liveness kernels.
    unsigned long long live_stream = 0;
    cudaEvent_t ev_pre = nullptr;
    // The operand tables of the verify kernels (vreg per operand, first-occurrence bits, table
    // offsets, vreg descriptors, first definitions) depend on the program alone: they are made by the
    // first liveness run and kept (layout arena).
    bool tables_built = false;

    // per-call working memory of vl_verify (one set per internal stream slot), grown on demand
    struct VScratch {
        void *block = nullptr;       // the allocation that holds the arrays below
        uint16_t *tg = nullptr;      // [groups][V+1][64] tables, 64 candidates side by side
        uint32_t *cstate = nullptr;  // [rows][8]
        uint32_t *anom = nullptr;    // [rows][AW] chunks whose walk collided
        uint32_t *work = nullptr;    // count, then items of the exact count: candidate, part | parts << 8
        uint32_t *racc = nullptr;    // [rows][4] accumulators of the exact count
        unsigned char *exact = nullptr;  // block arrays of the exact count that do not fit a multiprocessor
        uint32_t *grp_done = nullptr;  // walk thread blocks that have finished, per group of 64 candidates; then the groups' mark flags
        uint32_t *thm = nullptr;       // [groups][n_blocks][mask words][2][32] through-set masks
        uint64_t rows = 0, aw = 0, vregs = 0, chunks = 0;
    } vs[VL_LANES + 2];              // one per lane, then one per staging buffer of vl_verify_host
    VScratch fs[VL_LANES + 2];       // the same for what k_fused and k_eight hand to k_exact: cstate, anom, racc and (in work) the rows' items
    uint32_t sub_batch = 5120;       // candidates per pass of the verify kernels
    uint32_t lanes_opt = 3;          // lanes in use (1 = everything in order on the caller's stream)
    uint64_t lane_call = 0, lane_base = 0;  // the last vl_verify* call that spread passes over lanes, the lane of its first
    cudaEvent_t ev_fork = nullptr, ev_join[VL_LANES] = {};

    // opt-in per-kernel timing of vl_verify: five events per pass (before each of the four kernels, after the last)
    int ktime = 0;
    std::vector<cudaEvent_t> kt_ev;
    size_t kt_used = 0;

    // staging for vl_verify_host
    uint16_t *d_stage[2] = {nullptr, nullptr};
    vl_verdict *d_stage_out[2] = {nullptr, nullptr};
    uint64_t stage_rows = 0, stage_pitch = 0;
    vl_verdict *h_out_pinned = nullptr;  // verdicts of a vl_verify_host call on their way back
    uint64_t h_out_cap = 0;
    cudaStream_t h_streams[2] = {nullptr, nullptr};
    cudaEvent_t h_events[2] = {nullptr, nullptr};
    // the record that vl_verify_until_pass polls for, in pinned memory
    unsigned long long *h_rs = nullptr, rs_seq = 0;
    unsigned long long *d_diag_T = nullptr;  // [V] scratch of vl_diagnose: (first occurrence << 16) | value
    unsigned long long *d_diag_n = nullptr;  // one counter: scratch of vl_occupied_masks
};

extern std::atomic<uint64_t> g_vl_launches;

// Programmatic dependent launch: a kernel's blocks may start while the kernel before it in the stream still runs; what
// they do before pdl_wait reads the program, its layout and operand tables only.  pdl_go lets the next kernel's blocks
// start as soon as every block of this one has.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A launch that may (overlap) start before the launch in front of it has finished.
template <typename... P, typename... A>
static inline cudaError_t launch_overlap(void (*kernel)(P...), dim3 grid, uint32_t threads, size_t smem, cudaStream_t st, bool overlap,
                                         const A &...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = threads; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = &at; cfg.numAttrs = overlap ? 1 : 0;
    g_vl_launches.fetch_add(1);
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Lets a kernel use that many bytes of dynamic shared memory: asked for once per device, in front of its first launch (asking
// makes the driver load a kernel, also one that the process never uses).
template <auto kernel, int bytes>
static inline cudaError_t allow_smem(int device)
{
    static std::atomic<bool> done[64];
    if (device >= 0 && device < 64 && done[device].load()) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && device >= 0 && device < 64) done[device].store(true);
    return e;
}

#define VL_CUDA(prog, call)                     \
    do {                                        \
        cudaError_t e__ = (call);               \
        if (e__ != cudaSuccess) {               \
            (prog)->last_cuda_error = (int)e__; \
            return VL_ERR_CUDA;                 \
        }                                       \
    } while (0)

int vl_liveness_impl(vl_program *const *progs, uint32_t n, const cudaStream_t *streams, uint32_t n_streams);
// The one-kernel verify path of short jobs (vl_fused.cu): whether a job of K rows takes it, whether it may share a
// launch with other programs' jobs, and one launch for n <= VL_FUSED_MANY jobs.
#define VL_FUSED_MANY 48
bool vl_fused_wanted(vl_program *p, uint64_t K, bool alone = true);  // alone: k_eight would take the job instead
// Entries of the short chunks (vreg and short chunk at whose beginning it is occupied) from which a program counts as one
// that occupies many.
#define FUSED_MANY_ENTRIES 49152u  // (measured at vl_fused_wanted)
bool vl_verify_takes(const vl_program *p);  // whether the verify path takes the program (vl_verify.cu)
// The one-kernel verify path with eight candidates per thread block (vl_eight.cu): whether it takes a program at all, whether
// it is the one for a job of K rows, whether the job may share a launch, and one launch for n <= VL_EIGHT_MANY jobs.
#define VL_EIGHT_MANY 48
bool vl_eight_takes(const vl_program *p);
bool vl_eight_wanted(vl_program *p, uint64_t K);
bool vl_eight_shares(vl_program *p, uint64_t K);
bool vl_eight_hands(vl_program *p, uint64_t rows);  // whether a job of its own leaves counts to k_exact, in a working set
int vl_eight_run(uint32_t n, vl_program *const *progs, const uint16_t *const *d_cand, const uint64_t *K, const uint64_t *pitch,
                 vl_verdict *const *d_out, cudaStream_t from, cudaStream_t st, bool dict, int slot);  // slot: working set, -1: none
bool vl_fused_shares(vl_program *p, uint64_t K);
int vl_fused_run(uint32_t n, vl_program *const *progs, const uint16_t *const *d_cand, const uint64_t *K, const uint64_t *pitch,
                 vl_verdict *const *d_out, cudaStream_t from, cudaStream_t st, bool dict, int slot);  // slot: working set, -1: none
// The exact counts of the batched kernels' listed candidates (k_exact, vl_fused.cu).
// A candidate is listed twice, in items of about EXACT_FINE_CHUNKS and of about EXACT_PART_CHUNKS chunks of the walk.  The
// fine ones are taken if each has a thread block of its own: 1,000 rows of 8,000 instructions of which 100 fail 77 us
// against 81 for the whole call, 777 of 11,317 with 39 failing 103.5 against 109.  Beyond that what an item costs before
// its first count weighs more: 350 of the 1,000 failing 95 us in fine items, 85.5 in coarse ones.
#define EXACT_HDR 4         // words in front of the fine items, then the coarse ones: numbers of coarse and of fine items
#define EXACT_MAX_PARTS 32  // items of one candidate, at most
#define EXACT_MANY_PARTS 128  // the same of fine items, for programs that occupy many vregs (FUSED_MANY_ENTRIES): one row of 24,300
                              // instructions with 300 vregs live everywhere 0.56 ms, 1.23 with 32 items
#define EXACT_PART_CHUNKS 6
#define EXACT_FINE_CHUNKS 2
#define EXACT_FINE_ITEMS 512
#define EXACT_LONG 1024      // entries of an instruction's short list, on average, from which a warp counts them together
// per-candidate state between the kernels (8 words)
enum { CS_FLAGS = 0, CS_FIRST = 1, CS_BANK = 2, CS_WALK = 6, CS_THCOL = 7 };
enum : uint32_t { WALK_ANOM = 1u, WALK_FULL = 2u };
// Items of a candidate with that many chunks to count.
__device__ __forceinline__ uint32_t exact_parts(uint32_t chunks, uint32_t per_item, uint32_t most = EXACT_MAX_PARTS)
{
    return min(1u + chunks / per_item, most);
}
// Lists candidate k; fine_most: fine items of one candidate, at most.
__device__ __forceinline__ void list_exact(uint32_t *work, uint64_t k, uint32_t chunks, uint32_t fine_most)
{
    const uint32_t parts = exact_parts(chunks, EXACT_PART_CHUNKS), fine = exact_parts(chunks, EXACT_FINE_CHUNKS, fine_most);
    const uint32_t at = EXACT_FINE_ITEMS + atomicAdd(work, parts), fine_at = atomicAdd(work + 1, fine);
    for (uint32_t j = 0; j < parts; ++j) {
        work[EXACT_HDR + 2 * (at + j)] = (uint32_t)k;
        work[EXACT_HDR + 2 * (at + j) + 1] = j | (parts << 8);
    }
    for (uint32_t j = 0; j < fine && fine_at + j < EXACT_FINE_ITEMS; ++j) {
        work[EXACT_HDR + 2 * (fine_at + j)] = (uint32_t)k;
        work[EXACT_HDR + 2 * (fine_at + j) + 1] = j | (fine << 8);
    }
}
struct VlExactArgs {
    uint32_t *work, *cstate, *anom;
    const uint32_t *short_chunk, *chunk_short_off;  // [nS] chunk of every short chunk, [nC + 1] first short chunk of every chunk
    uint32_t *racc;               // [rows][4] overlaps, complement of the lowest instruction, bank tally, parts done; all 0
    uint32_t AW, nC, fine_items;      // fine_items: up to that many fine items are taken
    uint32_t rows;                // rows of k_fused or k_eight; 0: the candidates are listed in work
    uint32_t *items;              // [rows] a row's items, coarse | fine << 16
    uint32_t exact_bank;          // and an exact bank tally (k_fused)
    unsigned char *scratch;       // vl_exact_scratch bytes, null if 0
};
int vl_hand_scratch(vl_program *p, int slot, uint64_t rows, VlExactArgs *ex);  // what k_fused or k_eight share with k_exact
uint32_t vl_exact_blocks(vl_program *p);  // thread blocks of k_exact: one item each at a time
uint64_t vl_exact_scratch(vl_program *p);
bool vl_exact_takes_rows(vl_program *p, uint64_t rows);  // whether k_exact can count for that many rows of k_fused
int vl_exact_run(vl_program *p, const VlExactArgs &ex, const uint16_t *d_cand, uint64_t pitch, vl_verdict *d_out, cudaStream_t st,
                 bool dict, bool overlap);
// Records the next timing event of the handle on `st` (no-op unless kernel timing is switched on).
void kt_mark(vl_program *p, cudaStream_t st);
int vl_verify_impl(vl_program *p, const uint16_t *d_cand, uint64_t K, uint64_t pitch, vl_verdict *d_out,
                   cudaStream_t st, int slot, bool dict = false);
int vl_verify_lanes(uint32_t nprog, vl_program *const *progs, const uint16_t *const *d_cand, const uint64_t *K,
                    const uint64_t *pitch, vl_verdict *const *d_out, cudaStream_t st, bool dict = false);
// The lane streams of the handle's device (created once per device; the liveness stream
// follows the VL_LANES lanes in the array) and the handle's fork / join events.
int vl_lane_streams(vl_program *p, cudaStream_t **lanes);
void vl_free_liveness(vl_program *p);
// 128 bytes of pinned host memory, all zero (a pinned allocation of its own takes 155 us); null if there is none.
void *vl_pinned_get();
void vl_pinned_put(void *slot);
// Waits for a liveness run that is still in flight and checks its outcome; VL_OK if none is pending.
int vl_live_settle(vl_program *p);
// st waits for the liveness run in flight, if any; from: the stream that st's work of this call was forked from, or st.
int vl_live_join(vl_program *p, cudaStream_t from, cudaStream_t st);
// Multiprocessors of a device / of the handle's device (asked once).
int vl_device_sm_count(int device);
int vl_sm_count(vl_program *p);
