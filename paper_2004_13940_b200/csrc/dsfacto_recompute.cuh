// The recompute pass of the DS-FACTO epoch for sm_100a: auxiliaries, scores, multipliers, and the fp64 sums behind
// the objective.
#pragma once
#include <type_traits>

#include "dsfacto_common.cuh"
#include "dsfacto_epoch.cuh"

namespace dsf {

// ------------------------------------------------------------------------------------------
// Recompute pass (eq. (compute_a_jk), eq. (fm_model2), multiplier G).
//   a_ik = sum_j v_jk x_ij ; lin_i = sum_j w_j x_ij ; q_i = sum_j sum_k (v_jk x_ij)^2
//   f_i = w0 + lin_i + 1/2 (sum_k a_ik^2 - q_i)
// q_i is taken as sum_j x_ij^2 s_j with s_j = sum_k v_jk^2, which is the same sum regrouped: s_j is computed
// once per column after the parameters changed (model_view_kernel) and sits next to w_j, so the lane that
// owns an entry gets both with one 8-byte load and the K-wide part of an entry is K multiply-adds.
// MODE kScore: writes f only.  kTrain: writes A, G and per-CTA fp64 partial sums {sum l_i, sum G_i}.
// kEvaluate (held-out rows with labels; the quantities of the convergence figures of Section 5):
// writes nothing per row, per-CTA fp64 partial sums {sum l_i, sum t_i} with t_i = (f_i - y_i)^2 for
// the squared loss (RMSE) and t_i = [y_i f_i > 0] for the logistic loss (accuracy).
// kPartial (a handle that owns only a range of columns, Section 4.2's column blocks spread over
// workers): the sums run over the handle's own columns, so they are partial; writes a_ik, lin_i and
// q_i per row and stops there.  The partial sums of all shards are added outside and finish_kernel
// turns the totals into f_i, l_i and G_i.
// ------------------------------------------------------------------------------------------
// kScoreSums (the entry point that allocates nothing): f and the sums {sum l_i, sum G_i}.
enum { kScore = 0, kTrain = 1, kEvaluate = 2, kPartial = 3, kScoreSums = 4 };
struct RefreshArgs {
    int64_t n;
    const int64_t *indptr;
    const int32_t *idx;
    const float *val;
    const float *y;
    const float2 *pair;  // per column (w_j, s_j = sum_k v_jk^2)
    const float *w;      // RAW: w instead of the pairs
    double *sums_out;    // kScoreSums
    const float *V;
    float *A;
    float *G;
    float *f_out;
    float *lin_out, *q_out;  // kPartial: per-row partial sums
    double *partials;  // 4 per CTA: the two sums of the mode, sum w_j^2, sum v_jk^2
    float w0;
    int loss;
    // the squared norms of eq. (fm_obj), shared out over the CTAs (kTrain; norm_d = 0: left out)
    const float *norm_w, *norm_V;
    int64_t norm_d, norm_v4;
    // end of the pass: the last CTA adds the partial sums up
    unsigned *done;        // CTAs that have delivered (zero between launches)
    EpochState *st;        // kTrain: w0 comes from here and the sums go here; NULL: w0 above
    Report *report;        // mapped host memory (NULL: not the end of an epoch)
    uint32_t number;       // ... the number of the report (kTrain: counted on the device)
    int first;             // kTrain: the first segment of an epoch (its times are set, not added)
    int *bad;              // caller rows that were checked on the device: no row is read if it is set (NULL: sound rows)
};

// Sums of the whole launch in a fixed order: true in the last CTA to get here, whose thread 0 holds them.
__device__ __forceinline__ bool last_cta_sum4(double (&s)[4], double *partials, unsigned *done) {
    __shared__ bool last;
    block_sum4(s);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int c = 0; c < 4; ++c) partials[4 * (size_t)blockIdx.x + c] = s[c];
        __threadfence();
        last = atomicInc(done, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
#pragma unroll
    for (int c = 0; c < 4; ++c) s[c] = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += kThreads)
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] += __ldcg(partials + 4 * (size_t)b + c);
    block_sum4(s);
    return true;
}

// loss of a row and dl/df, its multiplier
__device__ __forceinline__ void loss_and_multiplier(int loss, float f, float y, float &li, float &gi) {
    if (loss == 0) {
        gi = f - y;
        li = 0.5f * gi * gi;
    } else {
        const float m = y * f;
        li = fmaxf(-m, 0.f) + log1pf(expf(-fabsf(m)));
        gi = -y / (1.f + expf(m));
    }
}
// what a held-out row adds to the metric: (f - y)^2 for the RMSE, or whether the sign of the score is the class
__device__ __forceinline__ double held_out_measure(int loss, float f, float y, float gi) {
    return loss == 0 ? (double)gi * (double)gi : y * f > 0.f ? 1.0 : 0.0;
}

// The last thread of a kernel whose CTAs have all written their results (to memory of the host as well): thread 0
// of the last CTA to get here.
__device__ __forceinline__ bool last_thread(unsigned *done) {
    __syncthreads();
    if (threadIdx.x != 0) return false;
    __threadfence_system();
    return atomicInc(done, gridDim.x - 1) == gridDim.x - 1;
}

// A warp takes GW = 32 / LG consecutive rows at a time, one per lane group, and stays converged: the loop over the
// entries runs to the longest of the rows (an earlier form in which every group looped on its own took 9.3 warp
// instructions per entry of 128-byte rows, most of them for the masks and branches of the divergent groups).  A batch
// is B = LG * E entries of each row, every lane owns E of them: it takes their (w_j, s_j) and hands column and value
// to its group; entries are requested two batches ahead.  Factor rows are requested UB entries at a time, NB - 1 steps
// ahead of the multiply-adds.  Behind the end of a row x is 0, and nothing is requested (TRIM): the registers
// keep the factors of an earlier entry of the row, whose infinities are the row's own, or zeros.  (Repeating the row's last
// entry there found it in L1, but each repetition took the look-ups and the data of a request: recompute pass, us, repeating
// and not: 2.6 M entries of text in 128-byte rows 42.7 and 40.9, 30 M in 512-byte rows 926 and 894, 11.7 M of click logs in
// 32-byte rows 95.3 and 93.8, 390 M in 64-byte rows 2780 and 2760.  Training passes over 12 M entries of tables, text and click
// logs with 3 to 128 factors: time repeating over time not 0.98 to 1.15, but for 3 factors and rows of 1 to 12 entries 0.95.
// Without pairs (RAW) some widths repeat: see launch_score_loss.)
// RAW: no pairs are at hand (the entry point that allocates nothing): w_j from w, s_j from the row itself.
// What bounds it: the gathers.  A skeleton of nothing but them (rows of one length, no sums at the end; the best of several
// widths of lane groups and depths) takes 2.57 ms for 390 M entries of click logs in 64-byte rows where this kernel takes 2.76,
// 38 us for 2.6 M of text in 128-byte rows (41), 0.31 ms for 17 M in 256-byte rows (0.37 for a call without pairs), 0.84 ms for
// 30 M in 512-byte rows (0.89): 152, 69, 54 and 36 G rows/s, 9 to 19 TB/s of L1 and L2 hits together.
// Not kept (each against the version it was tried on): columns and values as records of 8 bytes (2.97 -> 3.35 ms per 390 M
// entries of click logs); the pairs of the 2048 most frequent columns in shared memory, which the L1 then lacks (2.95 ->
// 2.98 ms); 64-byte rows requested three steps ahead instead of one (2.93 -> 2.98 ms); rows taken longest first inside
// blocks of 256 (text 44 -> 42.5 us, but click logs 2.97 -> 3.09 ms); two or four resident CTAs for 128-byte rows (46 and
// 43 us); lane groups that go on to their next row on their own (text 42.7 -> 39.5 us, click logs 2.78 -> 3.15 ms); on the
// skeleton, row and pair in one record of 80 or 128 bytes (0.54 -> 0.72 to 0.92 ms), 32-byte loads (no faster), entries staged
// through shared memory (0.61), hot rows and pairs there (0.55 to 0.8), hot rows kept in L1 by load policy (10 to 50 % slower).
template <int LG, int NV>
struct RefreshCfg {
    static constexpr int GW = 32 / LG;
    static constexpr int E = LG == 1 ? 4 : LG <= 4 ? 2 : 1;                 // entries per lane and batch
    static constexpr int LANES = LG < 8 ? LG : 8;                           // lanes of a group that hold entries
    static constexpr int B = LANES * E;                                     // entries of a row per batch
    static constexpr int UB = (LG == 8 && NV == 1) || LG == 4 ? 2 : 1;      // entries whose rows are requested together
    static constexpr int S = B / UB;                                        // steps per batch
    static constexpr int NB = LG * NV >= 48 || LG == 1 || LG == 4 ? 2 : 4;         // sets of registers: NB - 1 steps are under way
    static_assert(S % NB == 0, "a step keeps its registers from batch to batch");
    static constexpr int CTAS = LG < 8 ? 4 : NV >= 4 ? 2 : 3;  // resident per SM (register cap)
    static constexpr int ROWS = kThreads / LG;                              // rows per CTA and round
};
// Rows of 512 bytes and more: whether 16 lanes take a row instead of 8.  With 16, a lane has half as much of a row on its way,
// so that three CTAs fit an SM instead of two, and requests of a row are half as many; with 8, a warp has half the
// instructions per entry.  A table of factors that one L1 holds is read as fast as instructions are issued, a larger one as
// fast as requests are answered.  Recompute pass, us, 8 and 16 lanes: 512-byte rows, 30 M entries over 131 k columns 978 and
// 926, 2.8 M over 50 k 128 and 119, 3.9 M over 117 k 134 and 130, 2 M over 300, 500 and 1000 columns 63 and 69, 78 and 79, 84 and 78; 1-KB rows, 7.5 M entries
// over 131 k columns 494 and 447; 768-byte rows 379 and 357.  (Batches of 16 entries instead of 8: 905 in the first case, but
// 140 and 79 with rows of 39 and 20 entries.)
inline bool wide_recompute_groups(int64_t d, int Kp) { return Kp >= 128 && d * Kp * (int64_t)sizeof(float) > ((int64_t)320 << 10); }
template <int LG, int NV, int MODE, bool RAW = false, bool TRIM = true>
__global__ void __launch_bounds__(kThreads, (RefreshCfg<LG, NV>::CTAS)) refresh_kernel(const RefreshArgs a) {
    typedef RefreshCfg<LG, NV> C;
    constexpr int GW = C::GW, E = C::E, B = C::B, LANES = C::LANES, UB = C::UB, S = C::S, NB = C::NB, KP4 = LG * NV;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const int g = threadIdx.x / LG, l = threadIdx.x % LG, gw = (threadIdx.x & 31) / LG;
    const float4 *V4 = reinterpret_cast<const float4 *>(a.V) + l;
    float4 *A4 = reinterpret_cast<float4 *>(a.A);
    constexpr bool TRAIN = MODE == kTrain;
    constexpr bool STORE_A = MODE == kTrain || MODE == kPartial;
    // the fp64 sums of a lane group live in shared memory: only its first lane touches them, once per row
    __shared__ double sums[2][C::ROWS];
    if (l == 0) { sums[0][g] = 0.0; sums[1][g] = 0.0; }
    let_next_kernel_start();

    int64_t n = a.n;
    int bad = 0;
    if ((MODE == kScore || MODE == kEvaluate) && a.bad) {
        wait_for_previous_kernel();
        bad = *(volatile int *)a.bad;
        if (bad) n = 0;
    }
    const int64_t step = (int64_t)gridDim.x * C::ROWS;
    int64_t base = ((int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * GW;   // first row of the warp's set
    int64_t nbeg = 0;      // this group's row of the next set: its first entry and its length (at most d < 2^31)
    int nlen = 0;
    int32_t j0[E], j1[E], jn[E];   // entries of the batch at work, of the next one, of the next rows' first one
    float x0[E], x1[E], xn[E];
    auto next_pointers = [&](int64_t row) {
        nlen = 0;
        if (row < n) {
            nbeg = __ldg(a.indptr + row);
            nlen = (int)(__ldg(a.indptr + row + 1) - nbeg);
        }
    };
    auto load_entries = [&](int64_t beg, int t0, int len, int32_t (&j)[E], float (&x)[E]) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int t = t0 + e * LG + l;
            j[e] = TRIM ? -1 : 0; x[e] = 0.f;
            if (l >= LANES) continue;
            if (!TRIM && len > 0) j[e] = __ldg(a.idx + beg + min(t, len - 1));
            if (TRIM && t < len) j[e] = __ldg(a.idx + beg + t);
            if (t < len) x[e] = __ldg(a.val + beg + t);
        }
    };
    next_pointers(base + gw);
    load_entries(nbeg, 0, nlen, jn, xn);
    // (the rows do not change during an epoch; the model, which the kernel before this one writes, is read with
    // plain loads: the read-only path assumes data that nobody writes during the whole life of a kernel)
    wait_for_previous_kernel();
    if (TRAIN && a.st && blockIdx.x == 0 && threadIdx.x == 0) a.st->t1 = device_ns();
    const float w0 = TRAIN && a.st ? a.st->w0 : a.w0;
    for (; base < n; base += step) {
        const int64_t row = base + gw, beg = nbeg;
        const int len = nlen;
        next_pointers(row + step);
        const int longest = __reduce_max_sync(FULL, len);
        float4 acc[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        float q = 0.f, lin = 0.f;
        float2 q2 = make_float2(0.f, 0.f);   // (RAW)
        float4 vv[NB][UB][NV];
        auto load_rows = [&](const int32_t (&j)[E], int u0, float4 (&r)[UB][NV]) {
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int32_t ju = __shfl_sync(FULL, j[(u0 + u) / LG], (u0 + u) % LG, LG);
#pragma unroll
                for (int v = 0; v < NV; ++v)
                    if (!TRIM || ju >= 0) r[u][v] = V4[(size_t)ju * KP4 + v * LG];
            }
        };
#pragma unroll
        for (int e = 0; e < E; ++e) { j0[e] = jn[e]; x0[e] = xn[e]; }
        if (TRIM && len < NB * UB) {   // (no entry of this row will have been in every register by the time they are multiplied by zero)
#pragma unroll
            for (int st = 0; st < NB; ++st)
#pragma unroll
                for (int u = 0; u < UB; ++u)
#pragma unroll
                    for (int v = 0; v < NV; ++v) vv[st][u][v] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int st = 0; st + 1 < NB; ++st) load_rows(j0, st * UB, vv[st]);
        load_entries(beg, B, len, j1, x1);
        if (longest <= B) load_entries(nbeg, 0, nlen, jn, xn);
        for (int t0 = 0; t0 < longest; t0 += B) {
            int32_t j2[E];
            float x2[E];
            if (t0 + 2 * B < longest) load_entries(beg, t0 + 2 * B, len, j2, x2);
            else if (t0 + B < longest) load_entries(nbeg, 0, nlen, jn, xn);
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (l < LANES && t0 + e * LG + l < len) {
                    if (RAW) {
                        lin = fmaf(a.w[j0[e]], x0[e], lin);
                    } else {
                        const float2 ws = a.pair[j0[e]];
                        lin = fmaf(ws.x, x0[e], lin);
                        q = fmaf(x0[e] * x0[e], ws.y, q);
                    }
                }
#pragma unroll
            for (int st = 0; st < S; ++st) {
                const int ahead = st + NB - 1;
                if (ahead < S) load_rows(j0, ahead * UB, vv[ahead % NB]);
                else if (t0 + B < longest) load_rows(j1, (ahead - S) * UB, vv[ahead % NB]);
#pragma unroll
                for (int u = 0; u < UB; ++u) {
                    const float x = __shfl_sync(FULL, x0[(st * UB + u) / LG], (st * UB + u) % LG, LG);
                    const float4 (&r)[NV] = vv[st % NB][u];
#pragma unroll
                    for (int v = 0; v < NV; ++v) fma4(acc[v], x, r[v]);
                    if (RAW) {
                        float2 sv = make_float2(0.f, 0.f);
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            sv = __ffma2_rn(make_float2(r[v].x, r[v].y), make_float2(r[v].x, r[v].y), sv);
                            sv = __ffma2_rn(make_float2(r[v].z, r[v].w), make_float2(r[v].z, r[v].w), sv);
                        }
                        q2 = __ffma2_rn(sv, make_float2(x * x, x * x), q2);
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < E; ++e) { j0[e] = j1[e]; x0[e] = x1[e]; j1[e] = j2[e]; x1[e] = x2[e]; }
        }
        if (RAW) q = q2.x + q2.y;
        if (len == 0) {   // (a row without entries has added nothing but zeros times whatever row 0 holds)
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            q = 0.f;
        }
        float sq = 0.f;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            if (STORE_A && row < n) A4[(size_t)row * KP4 + v * LG + l] = acc[v];
            sq = fmaf(acc[v].x, acc[v].x, sq); sq = fmaf(acc[v].y, acc[v].y, sq);
            sq = fmaf(acc[v].z, acc[v].z, sq); sq = fmaf(acc[v].w, acc[v].w, sq);
        }
        if (MODE == kPartial) {
#pragma unroll
            for (int o = LG / 2; o > 0; o >>= 1) {
                q += __shfl_xor_sync(FULL, q, o);
                lin += __shfl_xor_sync(FULL, lin, o);
            }
            if (l == 0 && row < n) { a.lin_out[row] = lin; a.q_out[row] = q; }
            continue;
        }
        float pair = sq - q;
#pragma unroll
        for (int o = LG / 2; o > 0; o >>= 1) {
            pair += __shfl_xor_sync(FULL, pair, o);
            lin += __shfl_xor_sync(FULL, lin, o);
        }
        if (l == 0 && row < n) {
            const float f = w0 + lin + 0.5f * pair;
            if (MODE == kScore || MODE == kScoreSums) a.f_out[row] = f;
            if (MODE != kScore) {
                float li, gi;
                loss_and_multiplier(a.loss, f, a.y[row], li, gi);
                sums[0][g] += (double)li;
                if (TRAIN) a.G[row] = gi;
                sums[1][g] += TRAIN || MODE == kScoreSums ? (double)gi : held_out_measure(a.loss, f, a.y[row], gi);
            }
        }
    }
    if (MODE == kScore && last_thread(a.done)) {
        if (a.bad) *a.bad = 0;
        for (int i = 0; i < kReportWords<CallBody>; ++i) store_report_word(a.report->call + i, a.number, (uint32_t)bad);   // (nothing else is looked at)
    }
    if (MODE == kTrain || MODE == kEvaluate || MODE == kScoreSums) {
        double s[4] = {l == 0 ? sums[0][g] : 0.0, l == 0 ? sums[1][g] : 0.0, 0.0, 0.0};
        if (TRAIN) {
            const int64_t stride = (int64_t)gridDim.x * kThreads;
            for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < a.norm_d; i += stride) {
                const double x = (double)a.norm_w[i];
                s[2] += x * x;
            }
            const float4 *N4 = reinterpret_cast<const float4 *>(a.norm_V);
            for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < a.norm_v4; i += stride) {
                const float4 x = N4[i];
                s[3] += (double)x.x * x.x + (double)x.y * x.y + (double)x.z * x.z + (double)x.w * x.w;
            }
        }
        if (last_cta_sum4(s, a.partials, a.done) && threadIdx.x < 32) {
            __shared__ EpochBody ended;
            __shared__ CallBody called;
            uint32_t number = a.number;
            if (threadIdx.x == 0) {
                if (MODE == kScoreSums) { a.sums_out[0] = s[0]; a.sums_out[1] = s[1]; }
                if (MODE == kEvaluate) {
                    called.loss = s[0]; called.g = s[1]; called.bad = bad; called.unused = 0;
                    if (a.bad) *a.bad = 0;
                }
                if (TRAIN && a.st) {
                    EpochState &st = *a.st;
                    st.loss = s[0]; st.g = s[1]; st.w2 = s[2]; st.v2 = s[3];
                    const unsigned long long now = device_ns();
                    const unsigned long long ns0 = st.t1 - st.t0 + (a.first ? 0ull : st.ns[0]), ns1 = now - st.t1 + (a.first ? 0ull : st.ns[1]);
                    st.ns[0] = ns0; st.ns[1] = ns1;
                    if (a.report) {
                        ended.loss = s[0]; ended.g = s[1]; ended.w2 = s[2]; ended.v2 = s[3];
                        ended.w0 = st.w0;
                        ended.ns[0] = ns0; ended.ns[1] = ns1;
                        for (int c = 0; c < 3; ++c) ended.err[c] = st.err[c];
                        number = ++st.epochs;
                    }
                }
            }
            if (a.report && (MODE == kTrain || MODE == kEvaluate)) {
                number = __shfl_sync(0xFFFFFFFFu, number, 0);
                if (MODE == kTrain) store_report(a.report->epoch, number, ended);
                else store_report(a.report->call, number, called);
            }
        }
    }
}

}  // namespace dsf
