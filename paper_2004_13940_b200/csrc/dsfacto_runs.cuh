// Stratum SGD by column runs: the update loop of an epoch for data sets that are bucketed on the device.
//
// With G_i and a_i frozen the entries of a column, taken in the stratified order, map (w_j, v_j) affinely, and
// with D_T = prod_t (1 - e_t) - 1 (see dsfacto_sgd.cuh for the algebra)
//     v_j <- (1 + D_T) (v_j + U),   U = sum_t b_t / (1 + D_t) a_{i_t},
//     w_j <- (1 - ew)^T (w_j + W),  W = sum_t b_t (1 - ew)^{-t}.
// U, W and D_T do not depend on v_j, w_j, and pieces of a column combine by
//     U = U_1 + U_2 / (1 + D_1),  D = D_1 + D_2 + D_1 D_2,
// so nothing has to wait for anything: the entries of a pass are cut into equal units whatever the columns are,
// one warp per unit; a CTA joins the pieces of its warps, a second kernel (runs_apply_kernel) joins the few
// pieces of runs that cross CTAs and applies every run to its column once.
//
// Passes.  The rows are visited in the order row block p-1 .. 0, rows ascending inside a block, and cut into
// bands whose auxiliary rows stay in L2; one pass covers the entries of one band, sorted by (column, position in
// the stratified order).  A data set whose auxiliary rows fit L2 as a whole is one band: a column is then a
// single run in its full stratified order.  With several bands the entries of a column above its diagonal row
// block act on a tail composite q_j (same rule, started from zero, with its product kept in TS), folded in by
// runs_fold_kernel after the last band.  With the second schedule every segment has passes of its own.
#pragma once
#include "dsfacto_common.cuh"
#include "dsfacto_epoch.cuh"
#include "dsfacto_sgd.cuh"

namespace dsf {

constexpr int kRunWarps = 4;                      // warps (= units) per CTA of the sweep
constexpr int kRunThreads = 32 * kRunWarps;
constexpr int kUnitMax = 4096;                    // most entries of a unit
constexpr uint32_t kRunStart = 0x80000000u;       // bit of an entry's row word: first entry of a run

struct RunSweepArgs {
    const uint2 *ent;          // entries of the pass: {row | kRunStart, bits of x}
    int count;                 // their number
    int unit_len;              // entries per unit (a multiple of 32)
    const int *run_start;      // per run of the pass: its first entry
    const int *unit_run;       // per unit: the run that holds its first entry
    int nruns;
    int stamp;                 // first pass of a segment: note the time
    const float *A;            // n * Kp
    const float *G;            // n
    int64_t n;
    float4 *rec;               // per run: {D, W, -, -} and the K-wide sum
    float4 *part;              // per CTA: the piece of the run it found open, the piece of the run it left open
    EpochState *st;
    float h, lambda_v;
    float kappa_w;             // -log2(1 - ew)
};

#ifdef DSFACTO_DEBUG
#define DSF_RUN_CHECK(cond, code, value)                                                              \
    do {                                                                                              \
        if (!(cond) && atomicCAS(&a.st->err[0], 0, 3) == 0) { a.st->err[1] = (code); a.st->err[2] = (int)(value); } \
    } while (0)
#else
#define DSF_RUN_CHECK(cond, code, value) do { } while (0)
#endif

// lane layout of one warp: GW rows side by side, every lane group takes U consecutive entries of a stage
template <int LG, int NV>
struct RunCfg {
    static constexpr int GW = 32 / LG;
    static constexpr int KP4 = LG * NV;
    static constexpr int U = GW >= 8 ? 32 / GW : (NV >= 3 ? 2 : 4);
    static constexpr int ST = U * GW;        // entries per stage
    static constexpr int SP = 32 / ST;       // stages per pass of 32 entries
    static constexpr int REC = KP4 + 1;      // float4s of a record
    // CTAs of the sweep that stay resident per SM (register cap; the load cuts units by it).  More warps hide more of the
    // gathers until the registers for the rows on their way run out.  Update loops, us: 256-byte rows 4 / 5 / 6 CTAs (117 / 89 /
    // 76 registers), 2.6 M entries of text 78 / 71 / 72, 45 M in four bands 1045 / 975 / 944, 12 M of click logs 456 / 441 / 431,
    // 3 M over 300 columns 53 / 49 / 49; 64-byte rows 7 / 8 / 10, 390 M entries 4346 / 4089 / 5392; 128-byte rows 6 / 7, text
    // 40.9 / 43.8; 512-byte rows 4 / 5, 30 M entries 1227 / 1532.
    static constexpr int CTAS = KP4 <= 4 ? 8 : KP4 <= 16 ? 6 : 4;
};
template <int LG, int NV>
constexpr size_t run_sweep_smem() { return (size_t)kRunWarps * 2 * RunCfg<LG, NV>::REC * sizeof(float4); }

__device__ __forceinline__ float4 add4(const float4 a, const float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 zero4() { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ float4 shfl_xor4(const float4 x, int o) {
    return make_float4(__shfl_xor_sync(0xFFFFFFFFu, x.x, o), __shfl_xor_sync(0xFFFFFFFFu, x.y, o),
                       __shfl_xor_sync(0xFFFFFFFFu, x.z, o), __shfl_xor_sync(0xFFFFFFFFu, x.w, o));
}
__device__ __forceinline__ float4 shfl_up4(const float4 x, int o) {
    return make_float4(__shfl_up_sync(0xFFFFFFFFu, x.x, o), __shfl_up_sync(0xFFFFFFFFu, x.y, o),
                       __shfl_up_sync(0xFFFFFFFFu, x.z, o), __shfl_up_sync(0xFFFFFFFFu, x.w, o));
}
__device__ __forceinline__ float4 shfl_down4(const float4 x, int o) {
    return make_float4(__shfl_down_sync(0xFFFFFFFFu, x.x, o), __shfl_down_sync(0xFFFFFFFFu, x.y, o),
                       __shfl_down_sync(0xFFFFFFFFu, x.z, o), __shfl_down_sync(0xFFFFFFFFu, x.w, o));
}
__device__ __forceinline__ float4 shfl4(const float4 x, int from) {
    return make_float4(__shfl_sync(0xFFFFFFFFu, x.x, from), __shfl_sync(0xFFFFFFFFu, x.y, from),
                       __shfl_sync(0xFFFFFFFFu, x.z, from), __shfl_sync(0xFFFFFFFFu, x.w, from));
}
// the sum over the lane groups, in every group
template <int LG, int NV>
__device__ __forceinline__ void sum_groups(float4 (&x)[NV]) {
#pragma unroll
    for (int o = LG; o < 32; o <<= 1)
#pragma unroll
        for (int v = 0; v < NV; ++v) x[v] = add4(x[v], shfl_xor4(x[v], o));
}

// ------------------------------------------------------------------------------------------
// runs_sweep_kernel: one warp per unit of unit_len consecutive entries, walked in passes of 32.
//   scalar part   one entry per lane: G_i (requested one pass ahead) -> e, b; segmented scan of D = P - 1 over
//                 the lanes; coefficient c = b / P; the w coefficient.
//   K-wide part   a lane group of LG lanes takes U consecutive entries of a stage: their rows a_i go straight to
//                 registers (requested one stage ahead) and are added with weight c.  While no run ends, every
//                 group keeps its own partial sum; in a stage in which runs start, a group writes out the runs
//                 that lie inside it, and a segmented scan over the groups closes the others.
// A finished run goes to its record; the piece of the run that was open at the unit's start and the one left open
// at its end go to shared memory, where the CTA joins them.
// What bounds it (39 M entries of click logs, 64-byte rows, 365 us = 54 entries per clock of the GPU): the load / store
// data pipe is 79 % busy with 2.1 slots per entry: 0.68 shuffles and shared memory, 0.77 the gathered rows and words of
// G, the rest their look-ups.  L2 is at 62 % of its rate (a 64-byte row gather reaches 16 TB/s), instruction issue at
// 50 %.  A row ring that is copied from register to register (instead of requested into the registers that have just
// been used up) took 470 us; rows and coefficients handed to the groups through shared memory 365 us (a 16-byte
// broadcast load takes 2.05 slots); tile::gather4 copies reach 114 G rows/s against 250 G for plain loads.
// ------------------------------------------------------------------------------------------
template <int LG, int NV>
__global__ void __launch_bounds__(kRunThreads, (RunCfg<LG, NV>::CTAS)) runs_sweep_kernel(const RunSweepArgs a) {
    typedef RunCfg<LG, NV> C;
    constexpr int GW = C::GW, KP4 = C::KP4, U = C::U, ST = C::ST, SP = C::SP, REC = C::REC;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    extern __shared__ __align__(16) float4 pieces[];   // per warp: found open, left open
    __shared__ int s_seen[kRunWarps], s_ord[kRunWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane / LG, l = lane % LG;
    const int unit = blockIdx.x * kRunWarps + warp;
    const int base = unit * a.unit_len;
    const int len = min(a.unit_len, a.count - base);
    float4 *head = pieces + (size_t)warp * 2 * REC;
    for (int i = lane; i < REC; i += 32) head[i] = zero4();
    __syncwarp();
    let_next_kernel_start();

    bool seen = false;      // a run started in this unit
    int ord = 0;            // number of the run that is open
    if (len > 0) {
        const uint2 *ent = a.ent + base;
        auto load_entry = [&](int k) -> uint2 {
            const int at = 32 * k + lane;
            return at < len ? __ldcs(ent + at) : make_uint2(0u, 0u);
        };
        // entries and plan do not change during an epoch: they are requested before the wait for A and G
        const int npass = (len + 31) >> 5;
        uint2 e_c = load_entry(0), e_n = load_entry(1);
        ord = a.unit_run[unit];
        DSF_RUN_CHECK(ord >= 0 && ord < a.nruns, 20, ord);
        int run_begin = a.run_start[ord];
        if (__shfl_sync(FULL, e_c.x, 0) & kRunStart) ord -= 1;
        wait_for_previous_kernel();
        if (a.stamp && blockIdx.x == 0 && threadIdx.x == 0) a.st->t0 = device_ns();
        auto load_g = [&](const uint2 e, int k) -> float { return 32 * k + lane < len ? a.G[e.x & ~kRunStart] : 0.f; };
        const float4 *A4 = reinterpret_cast<const float4 *>(a.A) + l;
        // rows of a stage: with one stage per pass the next pass's rows are requested as soon as these are used up (the
        // scalar part of the next pass hides their latency), else the next stage's go to a second set of registers
        constexpr int NB = SP > 1 ? 2 : 1;
        float4 rows[NB][U][NV];
        auto load_rows = [&](const uint32_t row, int sp, float4 (&r)[U][NV]) {
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const uint32_t ir = __shfl_sync(FULL, row, sp * ST + g * U + i);
#pragma unroll
                for (int v = 0; v < NV; ++v) r[i][v] = A4[(size_t)ir * KP4 + v * LG];
            }
        };
        float g_c = load_g(e_c, 0);
        load_rows(e_c.x & ~kRunStart, 0, rows[0]);

        float4 acc[NV];        // this group's share of the open run's sum
#pragma unroll
        for (int v = 0; v < NV; ++v) acc[v] = zero4();
        float wl = 0.f;        // this lane's share of the open run's W
        float D_open = 0.f;    // product of the open run's entries in this unit, minus 1
        for (int k = 0; k < npass; ++k) {
            const uint2 e_f = load_entry(k + 2);
            const float g_n = load_g(e_n, k + 1);
            const uint32_t row_c = e_c.x & ~kRunStart, row_n = e_n.x & ~kRunStart;
            DSF_RUN_CHECK((int64_t)row_c < a.n, 21, row_c);
            const float x = __uint_as_float(e_c.y);
            const int cnt = min(32, len - 32 * k);
            const uint32_t mask = __ballot_sync(FULL, (e_c.x & kRunStart) != 0u);
            // ---- scalar part ----
            const float gx = g_c * x;
            const float b = -a.h * gx;
            float D = lane < cnt ? -a.h * (a.lambda_v - gx * x) : 0.f;
            float c;
            if (mask == 0u) {
#pragma unroll
                for (int delta = 1; delta < 32; delta <<= 1) {
                    const float up = __shfl_up_sync(FULL, D, delta);
                    if (lane >= delta) D = fmaf(up, D, up + D);
                }
                D = fmaf(D_open, D, D_open + D);
                c = b * rcp_fast(1.0f + D);
                wl = fmaf(b, ex2_fast((float)(base + 32 * k + lane + 1 - run_begin) * a.kappa_w), wl);
            } else {
                const uint32_t below = mask & (0xFFFFFFFFu >> (31 - lane));      // starts at or before this lane
                const int start = 31 - __clz(below);                                 // -1: the run was open before
                const int lim = below == 0u ? lane : lane - start;
                const int m = below == 0u ? base + 32 * k + lane + 1 - run_begin : lim + 1;
                const float cw = b * ex2_fast((float)m * a.kappa_w);
                float W_open = wl, W = cw;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) W_open += __shfl_xor_sync(FULL, W_open, o);
#pragma unroll
                for (int delta = 1; delta < 32; delta <<= 1) {
                    const float up = __shfl_up_sync(FULL, D, delta), upw = __shfl_up_sync(FULL, W, delta);
                    if (delta <= lim) { D = fmaf(up, D, up + D); W += upw; }
                }
                if (below == 0u) { D = fmaf(D_open, D, D_open + D); W += W_open; }
                c = b * rcp_fast(1.0f + D);
                // the last entry of a run that ends here leaves the run's product and W
                auto close = [&](int q, bool first, float d_, float w_) {
                    float2 *dst = reinterpret_cast<float2 *>(first ? head : a.rec + (size_t)q * REC);
                    DSF_RUN_CHECK(first || (q >= 0 && q < a.nruns), 22, q);
                    *dst = make_float2(d_, w_);
                };
                if (lane == 0 && (mask & 1u)) close(ord, !seen, D_open, W_open);
                if (lane < 31 && ((mask >> (lane + 1)) & 1u)) close(ord + __popc(below), below == 0u && !seen, D, W);
                const int last = 31 - __clz(mask);
                wl = lane >= last ? cw : 0.f;
                run_begin = base + 32 * k + last;
            }
            // ---- K-wide part ----
#pragma unroll
            for (int sp = 0; sp < SP; ++sp) {
                const float4 (&rw)[U][NV] = rows[sp % NB];
                if (SP > 1) {
                    if (sp + 1 < SP) load_rows(row_c, sp + 1, rows[(sp + 1) % NB]);
                    else load_rows(row_n, 0, rows[0]);
                }
                float cf[U];
#pragma unroll
                for (int i = 0; i < U; ++i) cf[i] = __shfl_sync(FULL, c, sp * ST + g * U + i);
                const uint32_t sub = ST == 32 ? mask : (mask >> (sp * ST)) & ((1u << (ST & 31)) - 1u);
                if (sub == 0u) {
#pragma unroll
                    for (int i = 0; i < U; ++i)
#pragma unroll
                        for (int v = 0; v < NV; ++v) fma4(acc[v], cf[i], rw[i][v]);
                } else {
                    sum_groups<LG, NV>(acc);   // what the stages before have of the open run; group 0 takes it along
                    if (g != 0) {
#pragma unroll
                        for (int v = 0; v < NV; ++v) acc[v] = zero4();
                    }
                    const uint32_t sb = (sub >> (g * U)) & ((1u << U) - 1u);
                    float4 lead[NV];           // this group's part of the run that ends at its first start
#pragma unroll
                    for (int v = 0; v < NV; ++v) lead[v] = zero4();
                    bool open = false;
#pragma unroll
                    for (int i = 0; i < U; ++i) {
                        if ((sb >> i) & 1u) {
                            if (!open) {
#pragma unroll
                                for (int v = 0; v < NV; ++v) lead[v] = acc[v];
                            } else {
                                const int pos = sp * ST + g * U + i;
                                float4 *dst = a.rec + (size_t)(ord + __popc(mask & ((1u << pos) - 1u))) * REC + 1 + l;
#pragma unroll
                                for (int v = 0; v < NV; ++v) dst[v * LG] = acc[v];
                            }
                            open = true;
#pragma unroll
                            for (int v = 0; v < NV; ++v) acc[v] = zero4();
                        }
#pragma unroll
                        for (int v = 0; v < NV; ++v) fma4(acc[v], cf[i], rw[i][v]);
                    }
                    // groups before this one, back to the last group with a start
                    const uint32_t upto = sub & (0xFFFFFFFFu >> (31 - (g * U + U - 1)));
                    const int lim = upto == 0u ? g : g - (31 - __clz(upto)) / U;
                    float4 t[NV];
#pragma unroll
                    for (int v = 0; v < NV; ++v) t[v] = acc[v];
#pragma unroll
                    for (int delta = 1; delta < GW; delta <<= 1)
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            const float4 up = shfl_up4(t[v], delta * LG);
                            if (delta <= lim) t[v] = add4(t[v], up);
                        }
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        float4 ex = shfl_up4(t[v], LG & 31);
                        if (g == 0) ex = zero4();
                        lead[v] = add4(lead[v], ex);
                    }
                    if (sb != 0u) {
                        const int pos = sp * ST + g * U + __ffs(sb) - 1;
                        const int before = __popc(mask & ((1u << pos) - 1u));
                        float4 *dst = (before == 0 && !seen ? head : a.rec + (size_t)(ord + before) * REC) + 1 + l;
#pragma unroll
                        for (int v = 0; v < NV; ++v) dst[v * LG] = lead[v];
                    }
                    if (g < (31 - __clz(sub)) / U) {   // summed into runs that have ended
#pragma unroll
                        for (int v = 0; v < NV; ++v) acc[v] = zero4();
                    }
                }
                if (SP == 1) load_rows(row_n, 0, rows[0]);
            }
            D_open = __shfl_sync(FULL, D, cnt - 1);
            if (mask != 0u) { seen = true; ord += __popc(mask); }
            e_c = e_n; e_n = e_f; g_c = g_n;
        }
        sum_groups<LG, NV>(acc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wl += __shfl_xor_sync(FULL, wl, o);
        float4 *dst = head + (seen ? REC : 0);
        if (g == 0) {
            if (l == 0) dst[0] = make_float4(D_open, wl, 0.f, 0.f);
#pragma unroll
            for (int v = 0; v < NV; ++v) dst[1 + v * LG + l] = acc[v];
        }
    } else {
        wait_for_previous_kernel();
        if (a.stamp && blockIdx.x == 0 && threadIdx.x == 0) a.st->t0 = device_ns();
    }
    if (lane == 0) { s_seen[warp] = seen ? 1 : 0; s_ord[warp] = ord; }
    __syncthreads();

    // ---- the CTA joins its warps' pieces in order, one float of the K-wide sum per thread ----
    for (int t = threadIdx.x; t < 4 * KP4; t += kRunThreads) {
        const int chunk = kRunWarps * a.unit_len;
        const int end = min(a.count, ((int)blockIdx.x + 1) * chunk);
        const bool ends_here = end == a.count || (a.ent[end].x & kRunStart) != 0u;
        float *part = reinterpret_cast<float *>(a.part + (size_t)blockIdx.x * 2 * REC);
        float *rec = reinterpret_cast<float *>(a.rec);
        float cu = 0.f, cd = 0.f, cw = 0.f;
        bool cs = false;     // the piece at hand belongs to a run that started in this CTA
        int co = 0;
        auto store = [&](float *dst) {
            dst[4 + t] = cu;
            if (t == 0) { dst[0] = cd; dst[1] = cw; }
        };
        for (int w = 0; w < kRunWarps; ++w) {
            const float *p = reinterpret_cast<const float *>(pieces + (size_t)w * 2 * REC);
            const float pd = p[0];
            cu = fmaf(p[4 + t], rcp_fast(1.0f + cd), cu);
            cw += p[1];
            cd = fmaf(cd, pd, cd + pd);
            if (s_seen[w]) {
                store(cs ? rec + (size_t)co * (4 * REC) : part);
                p += 4 * REC;
                cd = p[0]; cw = p[1]; cu = p[4 + t];
                cs = true;
                co = s_ord[w];
            }
        }
        store(!cs ? part : ends_here ? rec + (size_t)co * (4 * REC) : part + 4 * REC);
    }
}

// Position of an entry -> CTA of the sweep that has it: division by the CTA's entries, 128 k of them with k <= 128.
// q = p / 128 is below 2^24, so q / k = (q * ceil(2^32 / k)) >> 32 exactly (the inverse is too large by less than k / 2^32).
static_assert(kRunWarps * 32 == 128 && kUnitMax <= 128 * 32, "see chunk_of");
inline uint32_t chunk_inverse(int chunk) { return (uint32_t)((((uint64_t)1 << 32) + chunk / 128 - 1) / (uint64_t)(chunk / 128)); }   // (k = 1: 0)
__device__ __forceinline__ int chunk_of(int p, uint32_t inv) {
    const uint32_t q = (uint32_t)p >> 7;
    return (int)(inv == 0u ? q : __umulhi(q, inv));
}

struct RunApplyArgs {
    const uint32_t *run_key;   // per run: (column << 1) | acts on the tail composite
    const int *run_start;
    int nruns, count;          // runs and entries of the pass
    int chunk;                 // entries per CTA of the sweep
    uint32_t chunk_inv;        // chunk_inverse(chunk)
    const float4 *rec, *part;
    float *w, *V;
    float *Tw, *Tb;            // tail composite: q_j and its part for w (several bands only)
    float4 *TS;                // ... its product - 1 and its number of entries
    float2 *pair;              // per column (w_j, sum_k v_jk^2), where the recompute pass reads it; NULL: left to the fold
    float4 *Vs;                // copy of V in the recompute pass's column order, and ...
    const int32_t *slot_of;    // ... that order (NULL: pair is by column, no copy)
    EpochState *st;
    double w0_step;            // > 0: w0 takes its step, w0 -= w0_step * sum_i G_i
    double log1m_ew;           // log(1 - ew)
};

__device__ __noinline__ float pow_minus_1_wide(int m, double log1m_ew) { return (float)expm1((double)m * log1m_ew); }
// (1 - ew)^m - 1: a short series where that is exact to fp32, expm1 elsewhere
__device__ __forceinline__ float pow_minus_1(int m, double log1m_ew) {
    const float y = (float)m * (float)log1m_ew;
    if (fabsf(y) < 0.00390625f) return y * fmaf(y, fmaf(y, fmaf(y, 1.f / 24.f, 1.f / 6.f), 0.5f), 1.f);
    return pow_minus_1_wide(m, log1m_ew);
}

// ------------------------------------------------------------------------------------------
// runs_apply_kernel: every run of a pass acts on its column, once.  R runs per lane group, whose records and column
// rows are requested together (the kernel waits for memory most of the time: one run per group at a time left it
// at 1.3 TB/s), or one run per warp (COOP: few runs, each cut into many pieces).
// A run that lies in several CTAs of the sweep has a piece per CTA, and the most frequent column of a data set has dozens:
// joined one after the other by the run's own lane group they were a chain of that many trips to L2 (0.7 us each), behind
// which the kernel ended.  Rows of one float4 per lane: the whole warp joins them, a run at a time, also the two pieces of
// a run that only crosses a border (leaving those to the lane group costs registers).  Update loop, us, before and after:
// 2.6 M entries of 128-byte rows 46 -> 41, in four segments 96 -> 78, 11 M entries over 100 k columns 173 -> 152, 390 M
// entries of 64-byte rows 4300 -> 4130.  Wider rows keep the chain: the join takes registers with which two CTAs fit an SM
// instead of three (30 M entries of 512-byte rows in three bands 1240 -> 1263; 2.6 M in one band 125 -> 122).
// ------------------------------------------------------------------------------------------
template <int LG, int NV, bool COOP>
struct ApplyCfg {
    static constexpr int R = COOP ? 1 : 2;                         // runs per lane group
    static constexpr int RUNS = COOP ? kThreads / 32 : R * (kThreads / LG);      // runs per CTA
};
// Puts a piece behind the run's part (D, W, U) so far.
template <int NV>
__device__ __forceinline__ void join_piece(float &D, float &W, float4 (&U)[NV], float pd, float pw, const float4 (&x)[NV]) {
    const float inv = rcp_fast(1.0f + D);
#pragma unroll
    for (int v = 0; v < NV; ++v) fma4(U[v], inv, x[v]);
    W += pw;
    D = fmaf(D, pd, D + pd);
}
// The np pieces of the run that starts in CTA c0 of the sweep, by a whole warp: a lane group takes consecutive
// ones, AHEAD of them requested together, and a tree joins the groups' parts.  The whole is left in group 0.
template <int LG, int NV, int AHEAD>
__device__ __forceinline__ void join_pieces(const float4 *part, int c0, int np, float &D, float &W, float4 (&U)[NV]) {
    constexpr int GW = 32 / LG, REC = LG * NV + 1;
    const int lane = threadIdx.x & 31, l = lane % LG;
    const int per = (np + GW - 1) / GW, lo = min(np, lane / LG * per), hi = min(np, lo + per);
    D = 0.f; W = 0.f;
#pragma unroll
    for (int v = 0; v < NV; ++v) U[v] = zero4();
#pragma unroll(AHEAD)
    for (int i = lo; i < hi; ++i) {
        const float4 *p = part + ((size_t)(c0 + i) * 2 + (i == 0 ? 1 : 0)) * REC;
        const float4 hd = __ldcg(p);
        float4 x[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) x[v] = __ldcg(p + 1 + v * LG + l);
        join_piece<NV>(D, W, U, hd.x, hd.y, x);
    }
#pragma unroll
    for (int o = LG; o < 32; o <<= 1) {
        const float Do = __shfl_down_sync(0xFFFFFFFFu, D, o), Wo = __shfl_down_sync(0xFFFFFFFFu, W, o);
        float4 x[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) x[v] = shfl_down4(U[v], o);
        if (lane + o < 32) join_piece<NV>(D, W, U, Do, Wo, x);
    }
}
template <int LG, int NV, bool COOP>
__global__ void __launch_bounds__(kThreads, (NV == 1 ? 4 : 2)) runs_apply_kernel(const RunApplyArgs a) {
    constexpr int KP4 = LG * NV, REC = KP4 + 1;
    constexpr int R = ApplyCfg<LG, NV, COOP>::R, RUNS = ApplyCfg<LG, NV, COOP>::RUNS;
    constexpr unsigned FULL = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, l = lane % LG, g = lane / LG;
    let_next_kernel_start();
    int q[R], s[R], e[R];
    uint32_t key[R];
    int32_t slot[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int64_t id = (int64_t)blockIdx.x * RUNS + r * (RUNS / R) + threadIdx.x / (COOP ? 32 : LG);
        q[r] = id < a.nruns ? (int)id : -1;
        s[r] = 0; e[r] = 0; key[r] = 0u;
        if (q[r] >= 0) {
            s[r] = a.run_start[q[r]];
            e[r] = q[r] + 1 < a.nruns ? a.run_start[q[r] + 1] : a.count;
            key[r] = a.run_key[q[r]];
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) slot[r] = a.slot_of && q[r] >= 0 ? a.slot_of[key[r] >> 1] : (int32_t)(key[r] >> 1);
    wait_for_previous_kernel();
    if (a.w0_step > 0.0 && blockIdx.x == 0 && threadIdx.x == 0) a.st->w0 = (float)((double)a.st->w0 - a.w0_step * a.st->g);

    // ---- the column rows, and the records of the runs that lie in one CTA of the sweep ----
    float4 y[R][NV], U[R][NV];
    float D[R], W[R], yw[R];
    int np[R];
    auto row_of = [&](int r) { return reinterpret_cast<float4 *>((key[r] & 1u) ? a.Tb : a.V) + (int64_t)(key[r] >> 1) * KP4 + l; };
    auto w_of = [&](int r) { return ((key[r] & 1u) ? a.Tw : a.w) + (key[r] >> 1); };
#pragma unroll
    for (int r = 0; r < R; ++r) {
        np[r] = q[r] >= 0 ? chunk_of(e[r] - 1, a.chunk_inv) - chunk_of(s[r], a.chunk_inv) + 1 : 0;
        D[r] = 0.f; W[r] = 0.f; yw[r] = 0.f;
#pragma unroll
        for (int v = 0; v < NV; ++v) { y[r][v] = zero4(); U[r][v] = zero4(); }
        if (q[r] < 0) continue;
        if (!COOP || g == 0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) y[r][v] = __ldcg(row_of(r) + v * LG);
            if (l == 0) yw[r] = __ldcg(w_of(r));
        }
        if (np[r] == 1 ? !COOP || g == 0 : !COOP && NV > 1) {
            const float4 *p = np[r] == 1 ? a.rec + (size_t)q[r] * REC : a.part + ((size_t)chunk_of(s[r], a.chunk_inv) * 2 + 1) * REC;
            const float4 hd = __ldcg(p);
#pragma unroll
            for (int v = 0; v < NV; ++v) U[r][v] = __ldcg(p + 1 + v * LG + l);
            D[r] = hd.x; W[r] = hd.y;
        }
    }
    // ---- runs of several pieces: joined by the warp, one run after the other, or each by its own lane group ----
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int c0 = chunk_of(s[r], a.chunk_inv);
        if constexpr (!COOP && NV > 1) {
            for (int i = 1; i < np[r]; ++i) {
                const float4 *p = a.part + (size_t)(c0 + i) * 2 * REC;
                const float4 hd = __ldcg(p);
                float4 x[NV];
#pragma unroll
                for (int v = 0; v < NV; ++v) x[v] = __ldcg(p + 1 + v * LG + l);
                join_piece<NV>(D[r], W[r], U[r], hd.x, hd.y, x);
            }
        } else if constexpr (COOP) {
            if (np[r] > 1) join_pieces<LG, NV, 4>(a.part, c0, np[r], D[r], W[r], U[r]);
        } else {
            for (uint32_t todo = __ballot_sync(FULL, l == 0 && np[r] > 1); todo != 0u; todo &= todo - 1u) {
                const int owner = __ffs(todo) - 1;
                float Dr, Wr;
                float4 Ur[NV];
                join_pieces<LG, NV, 2>(a.part, __shfl_sync(FULL, c0, owner), __shfl_sync(FULL, np[r], owner), Dr, Wr, Ur);
                Dr = __shfl_sync(FULL, Dr, l);
                Wr = __shfl_sync(FULL, Wr, l);
#pragma unroll
                for (int v = 0; v < NV; ++v) Ur[v] = shfl4(Ur[v], l);
                if (g == owner / LG) {
                    D[r] = Dr; W[r] = Wr;
#pragma unroll
                    for (int v = 0; v < NV; ++v) U[r][v] = Ur[v];
                }
            }
        }
    }
    // ---- apply: y <- (1 + D) (y + U) ----
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const bool mine = q[r] >= 0 && (!COOP || g == 0);
        float sums[2] = {0.f, 0.f};   // of even and odd float4s: the order in which model_view_kernel adds
        if (mine) {
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                float4 t = add4(y[r][v], U[r][v]);
                t.x = fmaf(D[r], t.x, t.x); t.y = fmaf(D[r], t.y, t.y); t.z = fmaf(D[r], t.z, t.z); t.w = fmaf(D[r], t.w, t.w);
                row_of(r)[v * LG] = t;
                if (a.Vs) a.Vs[(int64_t)slot[r] * KP4 + v * LG + l] = t;
                float &sum = sums[v & 1];
                sum = fmaf(t.x, t.x, sum); sum = fmaf(t.y, t.y, sum); sum = fmaf(t.z, t.z, sum); sum = fmaf(t.w, t.w, sum);
            }
        }
        float sum = NV > 1 ? sums[0] + sums[1] : sums[0];
        if (a.pair) {
#pragma unroll
            for (int o = LG / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
        }
        if (mine && l == 0) {
            const float t = yw[r] + W[r];
            const int m = e[r] - s[r];
            const float wj = fmaf(pow_minus_1(m, a.log1m_ew), t, t);
            *w_of(r) = wj;
            if (a.pair) a.pair[slot[r]] = make_float2(wj, sum);
            if (key[r] & 1u) {
                const float4 ts = a.TS[key[r] >> 1];
                a.TS[key[r] >> 1] = make_float4(fmaf(ts.x, D[r], ts.x + D[r]), __int_as_float(__float_as_int(ts.y) + m), 0.f, 0.f);
            }
        }
    }
}

// After the last band of a segment: v_j <- (1 + D_T) v_j + q_j, w_j likewise, tail composites back to the
// identity, and the recompute pass's view of the model (pair, Vs) rebuilt.  A group of gs lanes per column.
__global__ void __launch_bounds__(kThreads) runs_fold_kernel(float4 *V, float *w, float4 *Tb, float *Tw, float4 *TS, int64_t d, int kp4,
                                                             int gs, const int32_t *slot_of, float4 *Vs, float2 *pair, double log1m_ew) {
    const int lane = (int)(threadIdx.x & 31u), gl = lane & (gs - 1);
    const int64_t groups = (int64_t)gridDim.x * (kThreads / gs);
    const int64_t g0 = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / gs;
    const int64_t rounds = (d + groups - 1) / groups;   // the same for every lane of a warp: the shuffles below stay converged
    let_next_kernel_start();
    wait_for_previous_kernel();
    for (int64_t it = 0; it < rounds; ++it) {
        const int64_t j = g0 + it * groups;
        float sums[2] = {0.f, 0.f};
        int64_t slot = j;
        float4 t = zero4();
        if (j < d) {
            if (slot_of) slot = slot_of[j];
            t = TS[j];
            const bool tail = __float_as_int(t.y) != 0;
            for (int v = gl; v < kp4; v += gs) {
                float4 y = V[j * kp4 + v];
                if (tail) {
                    const float4 q = Tb[j * kp4 + v];
                    y.x = fmaf(t.x, y.x, y.x) + q.x; y.y = fmaf(t.x, y.y, y.y) + q.y;
                    y.z = fmaf(t.x, y.z, y.z) + q.z; y.w = fmaf(t.x, y.w, y.w) + q.w;
                    V[j * kp4 + v] = y;
                    Tb[j * kp4 + v] = zero4();
                }
                if (Vs) Vs[slot * kp4 + v] = y;
                const bool odd = ((v / gs) & 1) != 0;
                float sum = odd ? sums[1] : sums[0];
                sum = fmaf(y.x, y.x, sum); sum = fmaf(y.y, y.y, sum); sum = fmaf(y.z, y.z, sum); sum = fmaf(y.w, y.w, sum);
                if (odd) sums[1] = sum; else sums[0] = sum;
            }
        }
        float sum = sums[0] + sums[1];
        for (int o = gs >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (j < d && gl == 0) {
            float wj = w[j];
            if (__float_as_int(t.y) != 0) {
                wj = fmaf(pow_minus_1(__float_as_int(t.y), log1m_ew), wj, wj) + Tw[j];
                w[j] = wj;
                Tw[j] = 0.f;
                TS[j] = zero4();
            }
            pair[slot] = make_float2(wj, sum);
        }
    }
}

// Start of an epoch (or of a recompute pass on its own) whose w0 the host has set.
__global__ void epoch_begin_kernel(EpochState *st, float w0) {
    st->w0 = w0;
    st->t0 = device_ns();
}

}  // namespace dsf
