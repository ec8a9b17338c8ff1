// Scores, or losses, of a small batch of rows that the host has laid out in mapped memory: a request.
#pragma once
#include "dsfacto_common.cuh"
#include "dsfacto_epoch.cuh"
#include "dsfacto_recompute.cuh"

namespace dsf {

// A request has the GPU to itself and lasts as long as its dependent steps: the launch, the trip across the link to the rows,
// the trip to the factor rows, the sums, the trip of the scores back.  So every row has a warp to itself, whose lane groups
// take its entries in turn and request the rows of a whole step (32 or 64 entries up to 256-byte rows) before they use the
// first; and the host lays the rows out in blocks, one per CTA, so that a CTA fetches what it needs, and no more, in one trip.
// Before, a lane group of the recompute kernel went through a row eight entries at a time (two trips to L2 for each eight),
// and either every CTA fetched the whole batch or each lane fetched its entries across the link, eight at a time.
// Calls of dsfacto_predict, K = 16, in us, before and after: 1 row of 39 entries 17.3 -> 12.7, 32 rows 21.6 -> 15.0, 300 rows
// 39.5 -> 31.0; 300 rows of one entry 19.0 -> 13.8, 5000 rows 33.5 -> 33.9; 1 row of 1000 entries 60 -> 28, of 8000 entries
// 1730 -> 130.  What bounds it: 8 us for a launch and its answer, 4 us in the interpreter, then the two trips.
constexpr int kMostBlockRows = 64;
// A block: first[block_rows + 1] (where the rows begin among the block's entries), then columns, values and labels.
struct RequestArgs {
    const uint4 *blocks;       // mapped host memory
    int stride;                // bytes from block to block (a multiple of 16)
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
};
template <int LG, int NV>
struct RequestCfg {
    static constexpr int GW = 32 / LG;
    static constexpr int UB = NV >= 6 ? 2 : NV == 4 ? 4 : LG == 1 ? 2 : LG == 2 ? 4 : 8;   // entries of a lane group per step
    static constexpr int STEP = GW * UB;                                                 // entries of a step
    static constexpr int E = STEP > 32 ? STEP / 32 : 1;                                  // ... per lane
};
template <int LG, int NV, int MODE>
__global__ void __launch_bounds__(kThreads) request_kernel(const RequestArgs a) {
    typedef RequestCfg<LG, NV> C;
    constexpr int GW = C::GW, UB = C::UB, STEP = C::STEP, E = C::E, KP4 = LG * NV;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    extern __shared__ __align__(16) uint4 block[];
    __shared__ float scores[kMostBlockRows];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % LG, g = lane / LG;
    let_next_kernel_start();
    const uint4 *from = a.blocks + (size_t)blockIdx.x * (a.stride / 16);
    constexpr int PIECES = 6;
    for (int i0 = threadIdx.x; i0 < a.stride / 16; i0 += PIECES * kThreads) {   // one trip across the link for up to 24 KB
        uint4 piece[PIECES];
#pragma unroll
        for (int i = 0; i < PIECES; ++i)
            if (i0 + i * kThreads < a.stride / 16) piece[i] = from[i0 + i * kThreads];
#pragma unroll
        for (int i = 0; i < PIECES; ++i)
            if (i0 + i * kThreads < a.stride / 16) block[i0 + i * kThreads] = piece[i];
    }
    __syncthreads();
    const int *first = reinterpret_cast<const int *>(block);
    const int entries = first[a.block_rows], rows = min(a.block_rows, a.rows - (int)blockIdx.x * a.block_rows);
    const int32_t *all_idx = first + a.block_rows + 1;
    const float4 *V4 = reinterpret_cast<const float4 *>(a.V) + l;
    wait_for_previous_kernel();   // the model

    for (int row = warp; row < rows; row += kThreads / 32) {
        const int beg = first[row], len = first[row + 1] - beg;
        const int32_t *idx = all_idx + beg;
        const float *val = reinterpret_cast<const float *>(idx + entries);
        float4 acc[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        float q = 0.f, lin = 0.f;
        for (int t0 = 0; t0 < len; t0 += STEP) {
            float4 r[UB][NV];
            float x[UB], xe[E];
            float2 ws[E];
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int t = t0 + u * GW + g;
                x[u] = 0.f;
#pragma unroll
                for (int v = 0; v < NV; ++v) r[u][v] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (t < len) {
                    x[u] = val[t];
#pragma unroll
                    for (int v = 0; v < NV; ++v) r[u][v] = V4[(size_t)idx[t] * KP4 + v * LG];
                }
            }
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int s = e * 32 + lane;
                xe[e] = 0.f; ws[e] = make_float2(0.f, 0.f);
                if (s < STEP && t0 + s < len) { xe[e] = val[t0 + s]; ws[e] = a.pair[idx[t0 + s]]; }
            }
#pragma unroll
            for (int u = 0; u < UB; ++u)
#pragma unroll
                for (int v = 0; v < NV; ++v) fma4(acc[v], x[u], r[u][v]);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                lin = fmaf(ws[e].x, xe[e], lin);
                q = fmaf(xe[e] * xe[e], ws[e].y, q);
            }
        }
#pragma unroll
        for (int o = LG; o < 32; o <<= 1)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                acc[v].x += __shfl_xor_sync(FULL, acc[v].x, o); acc[v].y += __shfl_xor_sync(FULL, acc[v].y, o);
                acc[v].z += __shfl_xor_sync(FULL, acc[v].z, o); acc[v].w += __shfl_xor_sync(FULL, acc[v].w, o);
            }
        float sq = 0.f;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            sq = fmaf(acc[v].x, acc[v].x, sq); sq = fmaf(acc[v].y, acc[v].y, sq);
            sq = fmaf(acc[v].z, acc[v].z, sq); sq = fmaf(acc[v].w, acc[v].w, sq);
        }
        float pair = g == 0 ? sq - q : -q;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
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
