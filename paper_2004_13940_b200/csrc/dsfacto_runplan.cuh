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
    const int32_t *col_start;
    int32_t per;               // rows that a warp takes at a time, at most 32
    uint32_t *key;
    unsigned long long *payload;
};

// floor(x / d) for x < 2^53 and d >= 1, with inv = 1 / d rounded: the product is off by less than one
__device__ __forceinline__ int64_t quotient(int64_t x, int64_t d, double inv) {
    int64_t q = (int64_t)((double)x * inv);
    const int64_t rest = x - q * d;
    return rest < 0 ? q - 1 : rest >= d ? q + 1 : q;
}
// A warp takes up to 32 rows at a time, a lane works out where each of them goes, and the warp walks their entries as one stretch,
// two windows of 32 at a time: the row of an entry is the number of row ends up to it (by bisection where rows are empty and
// ends coincide).  Divisions by n, d and the rows of a band are products with a correction, and in the plain schedule the
// phase of an entry is a comparison with the first column of its row's diagonal block.  (A warp per row with a 64-bit
// division per entry, 39 M entries: 437 us; now 180 us, 780 MB.)
__global__ void __launch_bounds__(kThreads) run_keys_kernel(const RunKeyArgs a) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t warp = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5, nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
    const double inv_n = 1.0 / (double)a.n, inv_d = 1.0 / (double)a.d, inv_band = 1.0 / (double)a.band_rows;
    const bool plain = a.every >= a.p;    // one segment
    for (int64_t i0 = a.per * warp; i0 < a.n; i0 += a.per * nwarps) {
        const int rows = (int)min((int64_t)a.per, a.n - i0);
        const int64_t i = i0 + min(lane, rows - 1);
        const int32_t r = (int32_t)quotient(i * (int64_t)a.p, a.n, inv_n);                  // row block
        const int64_t r0 = a.row_start[r], r1 = a.row_start[r + 1];
        const uint32_t band = (uint32_t)quotient((a.n - r1) + (i - r0), a.band_rows, inv_band);
        const uint32_t diagonal = (uint32_t)a.col_start[r];
        const int64_t beg = a.indptr[i], last = a.indptr[i + 1];
        const int64_t shift = (a.nnz - a.indptr[r1]) - a.indptr[r0];                        // place in visiting order, less the place in the CSR
        const int64_t from = __shfl_sync(FULL, beg, 0), to = __shfl_sync(FULL, last, 31);
        const int64_t end = lane < rows ? last : INT64_MAX;
        const bool holes = __any_sync(FULL, lane < rows && beg == last);
        auto place = [&](int64_t e0, uint32_t j, uint32_t x) {
            const int64_t e = e0 + lane, rel = end - e0;
            int k;                                                                          // rows that end at or before e
            if (holes) {
                k = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(FULL, end, k + step - 1) <= e) k += step;
            } else {
                const uint32_t ends = __reduce_or_sync(FULL, rel > 0 && rel < 32 ? 1u << (int)rel : 0u);
                k = __popc(__ballot_sync(FULL, rel <= 0)) + __popc(ends & ((2u << lane) - 1u));
            }
            k = min(k, 31);                                                                 // (behind the last entry)
            const int32_t rr = __shfl_sync(FULL, r, k);
            const uint32_t bb = __shfl_sync(FULL, band, k), dd = __shfl_sync(FULL, diagonal, k);
            const int64_t at = e + __shfl_sync(FULL, shift, k);
            if (e >= to) return;
            uint32_t pass = bb;
            bool tail = j < dd;                                                             // r > column block
            if (!plain) {
                const int32_t c = (int32_t)quotient((int64_t)j * a.p, a.d, inv_d);          // column block
                const int32_t seg = (c >= rr ? c - rr : c + a.p - rr) / a.every;            // of the round
                int32_t first = c - seg * a.every;                                          // the segment's first row block
                if (first < 0) first += a.p;
                pass += (uint32_t)seg * (uint32_t)a.bands;
                tail = rr > first;
            }
            a.key[at] = (((pass << a.cbits) | j) << 1) | (tail ? 1u : 0u);
            a.payload[at] = ((unsigned long long)x << 32) | (unsigned long long)(i0 + k);
        };
        for (int64_t e0 = from; e0 < to; e0 += 64) {
            uint32_t j[2], x[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int64_t e = e0 + 32 * u + lane;
                j[u] = e < to ? (uint32_t)a.idx[e] : 0u;
                x[u] = e < to ? __float_as_uint(a.val[e]) : 0u;
            }
            place(e0, j[0], x[0]);
            if (e0 + 32 < to) place(e0 + 32, j[1], x[1]);
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
// Which of a thread's eight consecutive entries start runs, and their keys: the passes over the sorted keys are as long as
// their requests are few and far between (one key and its predecessor at a time: 77 us per 39 M entries, now 28 us; the pass that writes the runs 132 -> 60 us).
constexpr int kKeysPerThread = kRunBlock / kThreads;
static_assert(kKeysPerThread == 8, "two 16-byte loads");
__device__ __forceinline__ uint32_t run_starts(const uint32_t *key, int64_t q0, int64_t nnz, int drop, uint32_t (&k)[kKeysPerThread]) {
    uint32_t before = 0u, starts = 0u;
    if (q0 + kKeysPerThread <= nnz) {   // (the array begins on a boundary of 256 bytes)
        const uint4 lo = *reinterpret_cast<const uint4 *>(key + q0), hi = *reinterpret_cast<const uint4 *>(key + q0 + 4);
        k[0] = lo.x; k[1] = lo.y; k[2] = lo.z; k[3] = lo.w; k[4] = hi.x; k[5] = hi.y; k[6] = hi.z; k[7] = hi.w;
    } else {
#pragma unroll
        for (int i = 0; i < kKeysPerThread; ++i) k[i] = q0 + i < nnz ? key[q0 + i] : 0u;
    }
    if (q0 > 0 && q0 < nnz) before = key[q0 - 1];
#pragma unroll
    for (int i = 0; i < kKeysPerThread; ++i) {
        const uint32_t prev = i == 0 ? before : k[i - 1];
        if (q0 + i < nnz && (q0 + i == 0 || (k[i] >> drop) != (prev >> drop))) starts |= 1u << i;
    }
    return starts;
}

// run starts per block of kRunBlock entries
__global__ void __launch_bounds__(kThreads) run_count_kernel(int64_t nnz, const uint32_t *__restrict__ key, int drop, int64_t *__restrict__ count) {
    __shared__ int total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    uint32_t k[kKeysPerThread];
    int mine = __popc(run_starts(key, (int64_t)blockIdx.x * kRunBlock + threadIdx.x * kKeysPerThread, nnz, drop, k));
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
    const int64_t q0 = (int64_t)blockIdx.x * kRunBlock + threadIdx.x * kKeysPerThread;
    uint32_t k[kKeysPerThread];
    const uint32_t starts = run_starts(a.key, q0, a.nnz, a.drop, k);
    const int mine = __popc(starts);
    int upto = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xFFFFFFFFu, upto, o);
        if (lane >= o) upto += up;
    }
    if (lane == 31) warp_sum[wid] = upto;
    __syncthreads();
    int64_t at = a.count[blockIdx.x] + (upto - mine);
    for (int w = 0; w < wid; ++w) at += warp_sum[w];
#pragma unroll
    for (int i = 0; i < kKeysPerThread; ++i) {
        if (((starts >> i) & 1u) == 0u) continue;
        a.ent[q0 + i].x |= kRunStart;
        a.run_start[at] = (int)(q0 + i - a.bounds[k[i] >> a.low_bits]);
        const uint32_t colphase = k[i] & ((2u << a.cbits) - 1u);
        a.run_key[at] = a.drop ? colphase & ~1u : colphase;
        ++at;
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

// Entries per column, from the runs of a pass: a few adds per column and none of them crowded.  (Counting the entries
// themselves takes as long as the adds to the most frequent columns take one after the other: 39 M entries 566 us, now 5 us.)
__global__ void __launch_bounds__(kThreads) run_columns_kernel(const int *__restrict__ run_start, const uint32_t *__restrict__ run_key, int nruns, int count,
                                                               int32_t *__restrict__ entries) {
    for (int64_t q = (int64_t)blockIdx.x * kThreads + threadIdx.x; q < nruns; q += (int64_t)gridDim.x * kThreads)   // (nearly 2^31 runs at most)
        atomicAdd(entries + (run_key[q] >> 1), (q + 1 < nruns ? run_start[q + 1] : count) - run_start[q]);
}

}  // namespace dsf
