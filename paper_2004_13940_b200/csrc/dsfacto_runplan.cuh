// Device side of dsfacto_load_csr for the update loop by column runs (dsfacto_runs.cuh): the stored entries in
// the order the passes read them, and the runs and units of every pass.
//   1. run_keys_kernel     per stored entry a 32-bit key (pass, column, phase) and a 64-bit payload (row, bits of
//                          x), written in visiting order: row block p-1 .. 0, rows ascending inside a block
//   2. a stable radix sort of the pairs by key (cub::DeviceRadixSort): inside a (pass, column) the visiting order
//      survives; the phase bit puts row blocks at or below the segment's first one in front, which makes it the
//      stratified order
//   3. pass_bounds_kernel  first entry of every pass (binary search in the sorted keys)
//   4. run_count_kernel / run_scan_kernel / run_write_kernel   the run starts: flagged in the entries, and listed
//      with their columns
//   5. unit_runs_kernel    per unit the run that holds its first entry
#pragma once
#include "dsfacto_common.cuh"
#include "dsfacto_runs.cuh"

namespace dsf {

constexpr int kRunBlock = 2048;   // entries per CTA of the passes over the sorted keys

struct RunKeyArgs {
    int64_t n, nnz;
    const int64_t *indptr;
    const int32_t *idx;
    const float *val;
    int32_t d, p;
    int cbits;                 // bits of a column index
    int64_t band_rows;         // rows per band, in visiting order
    int32_t bands;             // bands per segment
    int32_t every;             // rounds per segment
    const int64_t *row_start;
    uint32_t *key;
    unsigned long long *payload;
};

// One warp per row.
__global__ void __launch_bounds__(kThreads) run_keys_kernel(const RunKeyArgs a) {
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t warp = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
    for (int64_t i = warp; i < a.n; i += nwarps) {
        const int32_t r = (int32_t)(((uint64_t)i * (uint64_t)a.p) / (uint64_t)a.n);        // row block
        const int64_t r0 = a.row_start[r], r1 = a.row_start[r + 1];
        const uint32_t band = (uint32_t)(((a.n - r1) + (i - r0)) / a.band_rows);
        const int64_t beg = a.indptr[i], end = a.indptr[i + 1];
        int64_t out = (a.nnz - a.indptr[r1]) + (beg - a.indptr[r0]);
        for (int64_t e = beg + lane; e < end; e += 32) {
            const uint32_t j = (uint32_t)a.idx[e];
            const int32_t c = (int32_t)(((uint64_t)j * (uint64_t)a.p) / (uint64_t)a.d);     // column block
            const int32_t s = c >= r ? c - r : c + a.p - r;                                   // round
            const int32_t seg = s / a.every;
            int32_t first = c - seg * a.every;                                                // the segment's first row block
            if (first < 0) first += a.p;
            const uint32_t pass = (uint32_t)seg * (uint32_t)a.bands + band;
            const int64_t at = out + (e - beg);
            a.key[at] = (((pass << a.cbits) | j) << 1) | (r > first ? 1u : 0u);
            a.payload[at] = ((unsigned long long)__float_as_uint(a.val[e]) << 32) | (unsigned long long)i;
        }
    }
}

// bounds[q] = number of entries whose pass is below q, q = 0 .. npasses
__global__ void __launch_bounds__(kThreads) pass_bounds_kernel(int64_t nnz, const uint32_t *__restrict__ key, int low_bits, int npasses,
                                                               int64_t *__restrict__ bounds) {
    for (int q = blockIdx.x * kThreads + threadIdx.x; q <= npasses; q += gridDim.x * kThreads) {
        const uint64_t bound = (uint64_t)q << low_bits;
        int64_t lo = 0, hi = nnz;
        while (lo < hi) {
            const int64_t mid = lo + ((hi - lo) >> 1);
            if ((uint64_t)key[mid] < bound) lo = mid + 1; else hi = mid;
        }
        bounds[q] = lo;
    }
}

// drop: key bits that do not separate runs (1: the phase, when a column is one run in the whole segment)
__device__ __forceinline__ bool starts_run(const uint32_t *key, int64_t q, int drop) {
    return q == 0 || (key[q] >> drop) != (key[q - 1] >> drop);
}

// run starts per block of kRunBlock entries
__global__ void __launch_bounds__(kThreads) run_count_kernel(int64_t nnz, const uint32_t *__restrict__ key, int drop, int64_t *__restrict__ count) {
    __shared__ int total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    int mine = 0;
    for (int i = threadIdx.x; i < kRunBlock; i += kThreads) {
        const int64_t q = (int64_t)blockIdx.x * kRunBlock + i;
        if (q < nnz && starts_run(key, q, drop)) ++mine;
    }
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&total, mine);
    __syncthreads();
    if (threadIdx.x == 0) count[blockIdx.x] = total;
}

// exclusive prefix sum in place, the total behind the last element; one CTA
__global__ void __launch_bounds__(1024) run_scan_kernel(int64_t *count, int64_t blocks) {
    __shared__ int64_t warp_sum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t carry = 0;
    for (int64_t b0 = 0; b0 < blocks; b0 += 4096) {
        int64_t v[4], mine = 0;
        const int64_t at = b0 + (int64_t)threadIdx.x * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t c = at + i < blocks ? count[at + i] : 0;
            v[i] = mine;
            mine += c;
        }
        int64_t inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t up = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += up;
        }
        if (lane == 31) warp_sum[wid] = inc;
        __syncthreads();
        int64_t before = carry, all = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < wid) before += warp_sum[w];
            all += warp_sum[w];
        }
        before += inc - mine;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (at + i < blocks) count[at + i] = before + v[i];
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) count[blocks] = carry;
}

struct RunWriteArgs {
    int64_t nnz;
    const uint32_t *key;
    int drop, low_bits, cbits;
    const int64_t *count;      // run starts before each block
    const int64_t *bounds;     // first entry of every pass
    uint2 *ent;                // the sorted payloads: the run start bit is set here
    int *run_start;            // relative to the pass
    uint32_t *run_key;
};
__global__ void __launch_bounds__(kThreads) run_write_kernel(const RunWriteArgs a) {
    __shared__ int warp_sum[kThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int64_t at = a.count[blockIdx.x];
    for (int i0 = 0; i0 < kRunBlock; i0 += kThreads) {
        const int64_t q = (int64_t)blockIdx.x * kRunBlock + i0 + threadIdx.x;
        const bool st = q < a.nnz && starts_run(a.key, q, a.drop);
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, st);
        if (lane == 0) warp_sum[wid] = __popc(m);
        __syncthreads();
        int before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            if (w < wid) before += warp_sum[w];
            all += warp_sum[w];
        }
        if (st) {
            const int64_t k = at + before + __popc(m & ((1u << lane) - 1u));
            const uint32_t key = a.key[q];
            a.ent[q].x |= kRunStart;
            a.run_start[k] = (int)(q - a.bounds[key >> a.low_bits]);
            const uint32_t colphase = key & ((2u << a.cbits) - 1u);
            a.run_key[k] = a.drop ? colphase & ~1u : colphase;
        }
        at += all;
        __syncthreads();
    }
}

// first run of every pass: the number of run starts before its first entry
__global__ void __launch_bounds__(kThreads) pass_runs_kernel(int64_t nnz, const uint32_t *__restrict__ key, int drop, const int64_t *__restrict__ count,
                                                             int npasses, const int64_t *__restrict__ bounds, int64_t *__restrict__ run_first) {
    const int q = (blockIdx.x * kThreads + threadIdx.x) >> 5, lane = threadIdx.x & 31;   // one warp per pass
    if (q > npasses) return;
    const int64_t b = bounds[q], blk = b / kRunBlock;
    int mine = 0;
    for (int64_t e = blk * kRunBlock + lane; e < b; e += 32) mine += starts_run(key, e, drop) ? 1 : 0;
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if (lane == 0) run_first[q] = count[blk] + mine;
}

// per unit of a pass the run that holds its first entry (the last run that starts at or before it)
__global__ void __launch_bounds__(kThreads) unit_runs_kernel(const int *__restrict__ run_start, int nruns, int units, int unit_len,
                                                             int *__restrict__ unit_run) {
    for (int u = blockIdx.x * kThreads + threadIdx.x; u < units; u += gridDim.x * kThreads) {
        const int at = u * unit_len;
        int lo = 0, hi = nruns;   // first run that starts behind `at`
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (run_start[mid] <= at) lo = mid + 1; else hi = mid;
        }
        unit_run[u] = lo - 1;
    }
}

}  // namespace dsf
