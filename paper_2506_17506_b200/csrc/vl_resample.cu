// Statistics of the re-sampling loop over verdict arrays (Section 3.4, last paragraph: the model is
// sampled again until a candidate passes or the attempts run out; Section 4: Pass@k, AvgTry, MaxTry),
// and the loop itself in batches with early exit.
//
// Work per verdict: one 16-byte record read (coalesced, once); everything else is reductions.  For
// the row counts of the re-sampling loop (hundreds to tens of thousands of rows per test case) the
// kernels are launch-latency bound; a long array is spread over several thread blocks that combine
// with 64-bit atomics (minimum and sum: the result does not depend on their order).
#include "vl_internal.cuh"

namespace {

constexpr uint32_t RS_CASES = 96;     // test cases per launch (their pointers travel as kernel arguments)
constexpr uint32_t RS_THREADS = 512;
constexpr uint32_t RS_ROWS_PER_BLOCK = RS_THREADS * 16;  // a block takes about this many rows

struct RsParams {
    const uint4 *out[RS_CASES];  // verdict arrays
    uint64_t K[RS_CASES];
    vl_sample_stats *stats;      // [cases of this launch]
    uint32_t n;
};

__global__ void k_sample_init(const RsParams q)
{
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < q.n) { q.stats[c].first_pass = q.K[c]; q.stats[c].n_pass = 0; }
}

// grid (parts, cases): block (p, c) takes the rows p*T + t, (p + parts)*T + t, ... of case c
__global__ void __launch_bounds__(RS_THREADS) k_sample_stats(const RsParams q)
{
    const uint32_t c = blockIdx.y, tid = threadIdx.x;
    const uint64_t K = q.K[c];
    const uint64_t start = (uint64_t)blockIdx.x * RS_THREADS;
    if (start >= K && blockIdx.x) return;
    const uint4 *out = q.out[c];
    const uint64_t step = (uint64_t)gridDim.x * RS_THREADS;
    unsigned long long first = K, cnt = 0;
    for (uint64_t k = start + tid; k < K; k += step) {
        const uint4 v = __ldg(out + k);
        if (v.x & VL_PASS) {
            if (k < first) first = k;
            ++cnt;
        }
    }
#pragma unroll
    for (int d = 16; d; d >>= 1) {
        const unsigned long long f2 = __shfl_xor_sync(0xffffffffu, first, d);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, d);
        first = f2 < first ? f2 : first;
    }
    __shared__ unsigned long long s_first[RS_THREADS / 32], s_cnt[RS_THREADS / 32];
    if ((tid & 31) == 0) { s_first[tid >> 5] = first; s_cnt[tid >> 5] = cnt; }
    __syncthreads();
    if (tid == 0) {
        for (uint32_t w = 1; w < RS_THREADS / 32; ++w) {
            first = s_first[w] < first ? s_first[w] : first;
            cnt += s_cnt[w];
        }
        if (gridDim.x == 1) {  // one block per test case: nothing to combine with
            q.stats[c].first_pass = first;
            q.stats[c].n_pass = cnt;
        } else if (cnt) {
            atomicMin(reinterpret_cast<unsigned long long *>(&q.stats[c].first_pass), first);
            atomicAdd(reinterpret_cast<unsigned long long *>(&q.stats[c].n_pass), cnt);
        }
    }
}

struct RsSumParams {
    const vl_sample_stats *stats;
    vl_resample_summary *summary;
    uint32_t n, n_k;
    uint32_t k[VL_MAX_PASS_AT];
};

// one block: the records of all test cases -> the summary
__global__ void __launch_bounds__(256) k_resample_summary(const RsSumParams q)
{
    constexpr int N = 3 + VL_MAX_PASS_AT;  // solved, attempts summed, largest, pass@k
    __shared__ unsigned long long s[8][N];
    const uint32_t tid = threadIdx.x;
    unsigned long long v[N];
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = 0;
    pdl_wait();
    for (uint32_t c = tid; c < q.n; c += blockDim.x) {
        const vl_sample_stats r = q.stats[c];
        if (r.n_pass == 0) continue;
        const unsigned long long attempts = r.first_pass + 1;
        ++v[0];
        v[1] += attempts;
        v[2] = attempts > v[2] ? attempts : v[2];
#pragma unroll
        for (int j = 0; j < VL_MAX_PASS_AT; ++j)
            if ((uint32_t)j < q.n_k && attempts <= q.k[j]) ++v[3 + j];
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
#pragma unroll
        for (int d = 16; d; d >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, v[j], d);
            v[j] = j == 2 ? (o > v[j] ? o : v[j]) : v[j] + o;
        }
        if ((tid & 31) == 0) s[tid >> 5][j] = v[j];
    }
    __syncthreads();
    if (tid < N) {
        unsigned long long x = 0;
        for (int w = 0; w < 8; ++w) x = tid == 2 ? (s[w][tid] > x ? s[w][tid] : x) : x + s[w][tid];
        unsigned long long *out = tid < 3 ? (tid == 0 ? (unsigned long long *)&q.summary->n_solved
                                                      : (tid == 1 ? (unsigned long long *)&q.summary->sum_tries
                                                                  : (unsigned long long *)&q.summary->max_tries))
                                          : (unsigned long long *)&q.summary->pass_at[tid - 3];
        *out = x;
    }
    if (tid == 0) q.summary->n_cases = q.n;
}

// One block, the verdicts of a batch: its record goes straight to pinned host memory, then the sequence number that the host
// polls for (a kernel less, a copy less and no stream wait in the early-exit loop).  One block reads 5 verdicts per ns: 13 us
// in a loop of 109 for 4,096 rows of 64 instructions, 22 of 1,263 for 65,536, 78 of 7,403 for 400,000; the statistics kernels
// of many blocks, with their copy and wait, take 27, 29 and 46.
__global__ void __launch_bounds__(RS_THREADS) k_batch_record(const uint4 *out, uint32_t K, unsigned long long *record,
                                                             unsigned long long seq)
{
    __shared__ uint32_t s_first, s_cnt;
    if (threadIdx.x == 0) { s_first = K; s_cnt = 0; }
    __syncthreads();
    pdl_wait();
    uint32_t first = K, cnt = 0;
    for (uint32_t k = threadIdx.x; k < K; k += RS_THREADS)
        if (out[k].x & VL_PASS) { first = min(first, k); ++cnt; }
    first = __reduce_min_sync(0xffffffffu, first);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if ((threadIdx.x & 31) == 0 && cnt) { atomicMin(&s_first, first); atomicAdd(&s_cnt, cnt); }
    __syncthreads();
    if (threadIdx.x == 0) {
        record[0] = s_first;
        record[1] = s_cnt;
        __threadfence_system();
        *(volatile unsigned long long *)(record + 2) = seq;
    }
}

// records of cases [c0, c0 + m) into d_stats + c0
cudaError_t launch_stats(uint32_t m, const vl_verdict *const *d_out, const uint64_t *K, vl_sample_stats *d_stats,
                         cudaStream_t st, uint32_t max_parts)
{
    RsParams q;
    uint64_t kmax = 0;
    for (uint32_t j = 0; j < m; ++j) {
        q.out[j] = reinterpret_cast<const uint4 *>(d_out[j]);
        q.K[j] = K[j];
        kmax = K[j] > kmax ? K[j] : kmax;
    }
    q.stats = d_stats;
    q.n = m;
    uint64_t parts = (kmax + RS_ROWS_PER_BLOCK - 1) / RS_ROWS_PER_BLOCK;
    if (parts > max_parts) parts = max_parts;
    if (parts != 1) {  // (one block per test case writes its record itself)
        k_sample_init<<<1, RS_CASES, 0, st>>>(q);
        g_vl_launches.fetch_add(1);
    }
    if (kmax) {
        k_sample_stats<<<dim3((uint32_t)parts, m), RS_THREADS, 0, st>>>(q);
        g_vl_launches.fetch_add(1);
    }
    return cudaGetLastError();
}

}  // namespace

extern "C" int vl_resample_stats(int device, uint32_t n, const vl_verdict *const *d_out, const uint64_t *K,
                                 uint32_t n_k, const uint32_t *k, vl_sample_stats *d_stats,
                                 vl_resample_summary *d_summary, void *stream)
{
    if (n_k > VL_MAX_PASS_AT || (n_k && !k)) return VL_ERR_INVALID_ARG;
    if (n && (!d_out || !K || !d_stats)) return VL_ERR_INVALID_ARG;
    if (((uintptr_t)d_stats & 7) || ((uintptr_t)d_summary & 7)) return VL_ERR_INVALID_ARG;
    for (uint32_t j = 0; j < n; ++j)
        if (K[j] && (!d_out[j] || ((uintptr_t)d_out[j] & 15))) return VL_ERR_INVALID_ARG;
    if (n == 0 && !d_summary) return VL_OK;
    if (cudaSetDevice(device) != cudaSuccess) return VL_ERR_CUDA;
    cudaStream_t st = (cudaStream_t)stream;
    for (uint32_t c0 = 0; c0 < n; c0 += RS_CASES) {
        const uint32_t m = n - c0 < RS_CASES ? n - c0 : RS_CASES;
        // at most 4 thread blocks per multiprocessor work on one verdict array
        if (launch_stats(m, d_out + c0, K + c0, d_stats + c0, st, 4u * (uint32_t)vl_device_sm_count(device)) != cudaSuccess)
            return VL_ERR_CUDA;
    }
    if (d_summary) {
        RsSumParams s;
        s.stats = d_stats; s.summary = d_summary; s.n = n; s.n_k = n_k;
        for (uint32_t j = 0; j < VL_MAX_PASS_AT; ++j) s.k[j] = j < n_k ? k[j] : 0;
        if (launch_overlap(k_resample_summary, dim3(1), 256, 0, st, true, s) != cudaSuccess) return VL_ERR_CUDA;
    }
    return VL_OK;
}

extern "C" int vl_verify_until_pass(vl_program *p, const uint16_t *d_cand, uint64_t K, uint64_t pitch,
                                    uint64_t batch_rows, vl_verdict *d_out, uint64_t *rows_checked,
                                    uint64_t *first_pass, void *stream)
{
    if (!p || !rows_checked || !first_pass || batch_rows == 0) return VL_ERR_INVALID_ARG;
    *rows_checked = 0;
    *first_pass = K;
    if (!p->live_ok) return VL_ERR_LIVENESS_NOT_RUN;
    if (K == 0) return VL_OK;
    if (!d_cand || !d_out || ((uintptr_t)d_out & 15)) return VL_ERR_INVALID_ARG;
    VL_CUDA(p, cudaSetDevice(p->device));
    if (!p->h_rs && !(p->h_rs = (unsigned long long *)vl_pinned_get())) return VL_ERR_CUDA;
    volatile unsigned long long *rec = p->h_rs;  // first passing row, passing rows, sequence number
    cudaStream_t st = (cudaStream_t)stream;
    for (uint64_t b0 = 0; b0 < K; b0 += batch_rows) {
        const uint64_t nb = K - b0 < batch_rows ? K - b0 : batch_rows;
        const int rc = vl_verify(p, d_cand + b0 * pitch, nb, pitch, d_out + b0, stream);
        if (rc != VL_OK) return rc;
        const unsigned long long seq = ++p->rs_seq;
        VL_CUDA(p, launch_overlap(k_batch_record, dim3(1), RS_THREADS, 0, st, true, (const uint4 *)(d_out + b0), (uint32_t)nb,
                                  p->h_rs, seq));
        for (uint32_t polls = 0; rec[2] != seq;) {
            if (++polls < 4096) continue;
            polls = 0;
            const cudaError_t e = cudaStreamQuery(st);
            if (e == cudaErrorNotReady) continue;
            VL_CUDA(p, e);
            VL_CUDA(p, cudaStreamSynchronize(st));  // (finished: the record is there)
            if (rec[2] != seq) return VL_ERR_CUDA;
        }
        std::atomic_thread_fence(std::memory_order_acquire);
        *rows_checked = b0 + nb;
        if (rec[1]) {
            *first_pass = b0 + rec[0];
            break;
        }
    }
    return VL_OK;
}
