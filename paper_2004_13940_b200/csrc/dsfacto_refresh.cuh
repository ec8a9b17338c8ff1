// Kernels around the recompute pass (dsfacto_recompute.cuh): the view of the model it reads, the second half of a
// column shard's pass, the sums of the tile path's shards.
#pragma once
#include "dsfacto_common.cuh"
#include "dsfacto_recompute.cuh"

namespace dsf {

// Parameters of a small model to mapped host memory, with a report behind them.
__global__ void __launch_bounds__(kThreads) copy_out_kernel(const float *w, int64_t d, const float *V, int K, int Kp, float *out_w, float *out_V,
                                                            unsigned *done, Report *report, uint32_t number) {
    const int64_t stride = (int64_t)gridDim.x * kThreads, first = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    let_next_kernel_start();
    wait_for_previous_kernel();
    if (out_w)
        for (int64_t i = first; i < d; i += stride) out_w[i] = w[i];
    if (out_V)
        for (int64_t i = first; i < d * K; i += stride) out_V[i] = V[i / K * Kp + i % K];
    if (last_thread(done))
        for (int i = 0; i < kReportWords<CallBody>; ++i) store_report_word(report->call + i, number, 0u);
}

// ------------------------------------------------------------------------------------------
// Column slots for the recompute pass.  The pass gathers v_j and w_j by column index, and the L1 keeps
// whole 128-byte lines: with the columns where the data set put them, a hot 64-byte row shares its line
// with a cold neighbour and every hot w_j takes a line of its own.  The device copy of the CSR is
// therefore renumbered once per load, the most frequent column first (slot = rank by frequency: a count
// kernel, a stable radix sort of the d counters by cub::DeviceRadixSort, a rename kernel), and the
// pass reads a copy of V and of the pairs (w_j, s_j) in slot order: hot rows sit side by side, 16 hot pairs share one line.  The
// order of a row's entries does not change, so neither does any sum.  The stratum SGD kernels and
// everything a caller sees keep the column indices of the data set.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) column_count_kernel(const int32_t *__restrict__ idx, int64_t nnz, int32_t *__restrict__ count) {
    const int lane = (int)(threadIdx.x & 31u);
    // the loop bound is the same for all lanes of a warp, so the warp stays converged for the match
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; base < nnz; base += (int64_t)gridDim.x * blockDim.x) {
        const bool valid = base + lane < nnz;
        const int32_t j = valid ? idx[base + lane] : -1;
        // entries of the same column in one warp are counted by one lane
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, j);
        if (valid && lane == __ffs(peers) - 1) atomicAdd(count + j, __popc(peers));
    }
}
// sort key of a column: most frequent first (a column holds fewer than 2^31 entries); value: the column
__global__ void __launch_bounds__(kThreads) column_keys_kernel(const int32_t *__restrict__ count, int64_t d, uint32_t *__restrict__ key,
                                                               int32_t *__restrict__ column) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < d; j += (int64_t)gridDim.x * blockDim.x) {
        key[j] = 0x7FFFFFFFu - (uint32_t)count[j];
        column[j] = (int32_t)j;
    }
}
__global__ void __launch_bounds__(kThreads) column_slots_kernel(const int32_t *__restrict__ column_of, int64_t d, int32_t *__restrict__ slot_of) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < d; s += (int64_t)gridDim.x * blockDim.x)
        slot_of[column_of[s]] = (int32_t)s;
}
__global__ void __launch_bounds__(kThreads) column_rename_kernel(int32_t *__restrict__ idx, int64_t nnz, const int32_t *__restrict__ slot_of) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nnz; t += (int64_t)gridDim.x * blockDim.x)
        idx[t] = __ldg(slot_of + idx[t]);
}
// The model as the recompute pass reads it: pair[s] = (w_j, sum_k v_jk^2) and, when the columns are
// renumbered (column_of != NULL: j = column_of[s], and Vs is given), Vs[s] = V[j]; else j = s.  A group of gs
// lanes (a power of two <= 16) takes a row of kp4 float4s.
__global__ void __launch_bounds__(kThreads) model_view_kernel(const float4 *__restrict__ V, const float *__restrict__ w,
                                                              const int32_t *__restrict__ column_of, int64_t d, int kp4, int gs,
                                                              float4 *__restrict__ Vs, float2 *__restrict__ pair) {
    const int lane = (int)(threadIdx.x & 31u), gl = lane & (gs - 1);
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x / gs);
    const int64_t g0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / gs;
    const int64_t rounds = (d + groups - 1) / groups;   // the same for every lane of a warp: the shuffles below stay converged
    for (int64_t it = 0; it < rounds; ++it) {
        const int64_t s = g0 + it * groups;
        float sums[2] = {0.f, 0.f};   // of even and odd float4s of a lane (the tree over 32 lanes would start with these two)
        int64_t j = 0;
        if (s < d) {
            j = column_of ? (int64_t)__ldg(column_of + s) : s;
            for (int v = gl; v < kp4; v += gs) {
                const float4 x = V[j * kp4 + v];
                if (Vs) Vs[s * kp4 + v] = x;
                const bool odd = ((v / gs) & 1) != 0;
                float sum = odd ? sums[1] : sums[0];
                sum = fmaf(x.x, x.x, sum); sum = fmaf(x.y, x.y, sum); sum = fmaf(x.z, x.z, sum); sum = fmaf(x.w, x.w, sum);
                if (odd) sums[1] = sum; else sums[0] = sum;
            }
        }
        float sum = sums[0] + sums[1];
        for (int o = gs >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (s < d && gl == 0) pair[s] = make_float2(w[j], sum);
    }
}

// Second half of the recompute pass for column shards: from the summed auxiliaries a_i, lin_i, q_i of all
// shards to f_i = w0 + lin_i + 1/2 (sum_k a_ik^2 - q_i) (eq. (fm_model2)), the loss and the multiplier G_i;
// per-CTA fp64 partial sums {sum l_i, sum G_i}.  One lane group per row.
template <int LG, int NV>
__global__ void __launch_bounds__(kThreads) finish_kernel(int64_t n, const float *A, const float *lin, const float *q,
                                                          const float *y, float *G, double *partials, float w0, int loss) {
    constexpr int GR = kThreads / LG;
    constexpr int KP4 = LG * NV;
    const int g = threadIdx.x / LG, l = threadIdx.x % LG;
    const uint32_t gm = group_mask<LG>();
    const float4 *A4 = reinterpret_cast<const float4 *>(A);
    double loss_sum = 0.0, g_sum = 0.0;
    for (int64_t row = (int64_t)blockIdx.x * GR + g; row < n; row += (int64_t)gridDim.x * GR) {
        float sq = 0.f;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const float4 x = A4[(size_t)row * KP4 + v * LG + l];
            sq = fmaf(x.x, x.x, sq); sq = fmaf(x.y, x.y, sq); sq = fmaf(x.z, x.z, sq); sq = fmaf(x.w, x.w, sq);
        }
#pragma unroll
        for (int o = LG / 2; o > 0; o >>= 1) sq += __shfl_xor_sync(gm, sq, o, LG);
        if (l == 0) {
            const float f = w0 + lin[row] + 0.5f * (sq - q[row]);
            const float yy = y[row];
            float li, gi;
            if (loss == 0) {
                gi = f - yy;
                li = 0.5f * gi * gi;
            } else {
                const float m = yy * f;
                li = fmaxf(-m, 0.f) + log1pf(expf(-fabsf(m)));
                gi = -yy / (1.f + expf(m));
            }
            G[row] = gi;
            loss_sum += (double)li;
            g_sum += (double)gi;
        }
    }
    block_sum2(loss_sum, g_sum);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = loss_sum;
        partials[2 * blockIdx.x + 1] = g_sum;
    }
}

// per-CTA fp64 partial sums {sum w_j^2, sum v_jk^2}
__global__ void __launch_bounds__(kThreads) sqnorm_kernel(const float *w, int64_t d, const float *V, int64_t dkp,
                                                          double *partials) {
    double sw = 0.0, sv = 0.0;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < d; i += stride) {
        const double x = (double)w[i];
        sw += x * x;
    }
    const float4 *V4 = reinterpret_cast<const float4 *>(V);
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < dkp / 4; i += stride) {
        const float4 x = V4[i];
        sv += (double)x.x * x.x + (double)x.y * x.y + (double)x.z * x.z + (double)x.w * x.w;
    }
    block_sum2(sw, sv);
    if (threadIdx.x == 0) {
        partials[2 * blockIdx.x] = sw;
        partials[2 * blockIdx.x + 1] = sv;
    }
}

// out[c] = sum over CTAs b (ascending, fixed tree) of partials[2*b + c], c = 0,1
__global__ void __launch_bounds__(kThreads) reduce2_kernel(const double *partials, int nblocks, double *out) {
    double s0 = 0.0, s1 = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kThreads) {
        s0 += partials[2 * b];
        s1 += partials[2 * b + 1];
    }
    block_sum2(s0, s1);
    if (threadIdx.x == 0) { out[0] = s0; out[1] = s1; }
}

}  // namespace dsf
