// Scores, or losses, of a small batch of rows that the host has laid out in mapped memory: a request.
#pragma once
#include "dsfacto_common.cuh"
#include "dsfacto_epoch.cuh"
#include "dsfacto_recompute.cuh"
#include "dsfacto_request.h"

namespace dsf {

// A request has the GPU to itself and lasts as long as its dependent steps: the launch, the trip across the link to the rows,
// the trip to the factor rows, the sums, the trip of the scores back.  So every row has a warp to itself, which requests the
// factor rows of a whole step (64 entries of up to 128 bytes, 8 KB of wider ones) into shared memory before it uses the first;
// and the host lays the rows out in blocks, one per CTA, so that a CTA fetches what it needs, and no more, in one trip.
// The sums are those of the recompute kernel, bit for bit: a row scored on its own has the score it has among others.
// Before, a lane group of the recompute kernel went through a row eight entries at a time (two trips to L2 for each eight),
// and either every CTA fetched the whole batch or each lane fetched its entries across the link, eight at a time.
// Calls of dsfacto_predict, K = 16, in us, before and after: 1 row of 39 entries 17.3 -> 13.5, 32 rows 21.6 -> 15.7, 300 rows
// 39.5 -> 27.8; 300 rows of one entry 19.0 -> 13.6, 5000 rows 33.5 -> 31.7; 1 row of 1000 entries 60 -> 50, of 8000 entries
// 1730 -> 315.  What bounds it: 8 us for a launch and its answer, 4 us in the interpreter, then the two trips.  (Lane groups
// that each sum up a part of the row and add their parts at the end take 14.5 us for 32 rows, but round differently.)
struct RequestArgs {
    const uint4 *blocks;       // mapped host memory, laid out by lay_out_request
    int block_rows;            // rows of a block (at most kMostBlockRows)
    int rows;                  // of the batch
    const float2 *pair;        // per column (w_j, s_j = sum_k v_jk^2)
    const float *V;
    float w0;
    int loss;
    unsigned long long *f_words;   // kScore: the scores, in mapped host memory, as words of a report each
    Report *report;            // kEvaluate
    uint32_t number;           // of the words
    double *partials;          // kEvaluate: 4 per CTA
    unsigned *done;            // CTAs that have delivered (zero between launches)
    uint16_t at[kMostBlocks + 1];  // first word of every block, and the word behind the last one
};
template <int LG, int NV>
struct RequestCfg {
    static constexpr int KP4 = LG * NV;
    static constexpr int STEP = KP4 <= 8 ? 64 : (512 / KP4) & ~7;      // entries whose factor rows are on their way together: 8 KB at most
    static constexpr int F = (KP4 + 31) / 32;                          // float4s of a row per lane
};
// what a warp keeps in shared memory: the factor rows and the pairs (w_j, s_j) of a step
template <int LG, int NV>
struct RequestStep {
    float4 rows[RequestCfg<LG, NV>::STEP * RequestCfg<LG, NV>::KP4];
    float2 pairs[RequestCfg<LG, NV>::STEP];
};
template <int LG, int NV>
constexpr size_t request_smem(size_t largest_block) { return sizeof(RequestStep<LG, NV>) * (kThreads / 32) + largest_block; }
template <int LG, int NV, int MODE>
__global__ void __launch_bounds__(kThreads) request_kernel(const __grid_constant__ RequestArgs a) {
    typedef RequestCfg<LG, NV> C;
    constexpr int STEP = C::STEP, F = C::F, KP4 = C::KP4, LANES = RefreshCfg<LG, NV>::LANES;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    extern __shared__ __align__(16) uint4 shared[];
    RequestStep<LG, NV> &step = reinterpret_cast<RequestStep<LG, NV> *>(shared)[threadIdx.x >> 5];
    uint4 *block = shared + sizeof(RequestStep<LG, NV>) * (kThreads / 32) / 16;
    __shared__ float scores[kMostBlockRows];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % LG;
    let_next_kernel_start();
    const int word = a.at[blockIdx.x];                                          // the 16-byte units that hold the block
    const uint4 *from = a.blocks + word / 4;
    const int units = (a.at[blockIdx.x + 1] + 3) / 4 - word / 4;
    constexpr int PIECES = 6;
    for (int i0 = threadIdx.x; i0 < units; i0 += PIECES * kThreads) {           // one trip across the link for up to 24 KB
        uint4 piece[PIECES];
#pragma unroll
        for (int i = 0; i < PIECES; ++i)
            if (i0 + i * kThreads < units) piece[i] = from[i0 + i * kThreads];
#pragma unroll
        for (int i = 0; i < PIECES; ++i)
            if (i0 + i * kThreads < units) block[i0 + i * kThreads] = piece[i];
    }
    __syncthreads();
    const int *ends = reinterpret_cast<const int *>(block) + word % 4;
    const int rows = min(a.block_rows, a.rows - (int)blockIdx.x * a.block_rows), entries = ends[rows - 1];
    const int32_t *all_idx = ends + rows;
    const float4 *V4 = reinterpret_cast<const float4 *>(a.V);
    wait_for_previous_kernel();   // the model

    for (int row = warp; row < rows; row += kThreads / 32) {
        const int beg = row > 0 ? ends[row - 1] : 0, len = ends[row] - beg;
        const int32_t *idx = all_idx + beg;
        const float *val = reinterpret_cast<const float *>(idx + entries);
        float4 acc[F];
#pragma unroll
        for (int i = 0; i < F; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        float q = 0.f, lin = 0.f;
        for (int t0 = 0; t0 < len; t0 += STEP) {
            const int now = min(STEP, len - t0);
            for (int i = lane; i < now * KP4; i += 32) {
                const uint32_t to = (uint32_t)__cvta_generic_to_shared(step.rows + i);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(V4 + (size_t)idx[t0 + i / KP4] * KP4 + i % KP4) : "memory");
            }
            for (int t = lane; t < now; t += 32) step.pairs[t] = a.pair[idx[t0 + t]];
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
            // in the order of the entries, a lane one part (or two) of the row
#pragma unroll 8
            for (int t = 0; t < now; ++t) {
                const float x = val[t0 + t];
#pragma unroll
                for (int i = 0; i < F; ++i) fma4(acc[i], x, step.rows[t * KP4 + min(lane + 32 * i, KP4 - 1)]);
            }
            // ... and a lane the scalars of every eighth entry (or LG-th), as the recompute kernel does
#pragma unroll 4
            for (int t = l < LANES ? l : now; t < now; t += LANES) {
                const float x = val[t0 + t];
                const float2 ws = step.pairs[t];
                lin = fmaf(ws.x, x, lin);
                q = fmaf(x * x, ws.y, q);
            }
            __syncwarp();
        }
        float sq = 0.f;
#pragma unroll
        for (int v = 0; v < NV; ++v) {   // float4 number v * LG + l of the row
            const float4 y = acc[v * LG / 32];
            const int from = (v * LG + l) & 31;
            const float4 z = make_float4(__shfl_sync(FULL, y.x, from), __shfl_sync(FULL, y.y, from), __shfl_sync(FULL, y.z, from), __shfl_sync(FULL, y.w, from));
            sq = fmaf(z.x, z.x, sq); sq = fmaf(z.y, z.y, sq); sq = fmaf(z.z, z.z, sq); sq = fmaf(z.w, z.w, sq);
        }
        float pair = sq - q;
#pragma unroll
        for (int o = LG / 2; o > 0; o >>= 1) {
            pair += __shfl_xor_sync(FULL, pair, o);
            lin += __shfl_xor_sync(FULL, lin, o);
        }
        if (lane == 0) scores[row] = a.w0 + lin + 0.5f * pair;
    }
    __syncthreads();
    const int mine = threadIdx.x, row0 = (int)blockIdx.x * a.block_rows;
    if (MODE == kScore) {
        if (mine < rows) store_report_word(a.f_words + row0 + mine, a.number, __float_as_uint(scores[mine]));
        return;
    }
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    if (mine < rows) {
        const float f = scores[mine], y = reinterpret_cast<const float *>(all_idx + 2 * entries)[mine];
        float li, gi;
        loss_and_multiplier(a.loss, f, y, li, gi);
        s[0] = (double)li;
        s[1] = held_out_measure(a.loss, f, y, gi);
    }
    if (last_cta_sum4(s, a.partials, a.done) && warp == 0) {
        __shared__ CallBody called;
        if (lane == 0) { called.loss = s[0]; called.g = s[1]; called.bad = 0; called.unused = 0; }
        store_report(a.report->call, a.number, called);
    }
}

}  // namespace dsf
