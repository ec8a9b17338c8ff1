// Kernels around the training path: the seeded draw of V, the checks of caller data that is already on the
// device, and the change between the caller's factor rows (K floats) and the handle's (Kp floats).
#pragma once
#include "dsfacto_common.cuh"

namespace dsf {

// ---- SplitMix64 (Steele, Lea, Flood 2014), random access to the c-th output ----
__host__ __device__ inline uint64_t splitmix64_output(uint64_t seed, uint64_t c) {
    uint64_t z = seed + (c + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__host__ __device__ inline double open_unit(uint64_t u) { return ((double)(u >> 11) + 0.5) * (1.0 / 9007199254740992.0); }
// element e of the initial V before it is rounded to fp32 (Box-Muller, cosine branch)
__host__ __device__ inline double init_factor(uint64_t seed, uint64_t e) {
    const double u1 = open_unit(splitmix64_output(seed, 2 * e));
    const double u2 = open_unit(splitmix64_output(seed, 2 * e + 1));
    return 0.01 * (sqrt(-2.0 * log(u1)) * cos(2.0 * 3.14159265358979323846 * u2));
}

// The draw of V on the device (134 M factors: 0.47 s on 16 host cores, about a millisecond here).  The value
// handed out is the fp32 rounding of what the host's log and cos give; the device's may differ from them by a few
// ulps of fp64, which matters only if the value lies that close to the middle between two fp32 numbers.  Such
// elements (64 ulps to either side: one in four million) are listed, and the host recomputes them.
__global__ void __launch_bounds__(kThreads) init_factors_kernel(uint64_t seed, int64_t d, int K, int Kp, float *V, int *listed, int64_t *list, int most) {
    const int64_t total = d * Kp, stride = (int64_t)gridDim.x * kThreads;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < total; i += stride) {
        const int64_t j = i / Kp;
        const int k = (int)(i - j * Kp);
        float v = 0.f;
        if (k < K) {
            const double x = init_factor(seed, (uint64_t)(j * K + k));
            v = (float)x;
            const long long low = __double_as_longlong(x) & 0x1FFFFFFFll;   // mantissa bits fp32 has no room for
            if (llabs(low - 0x10000000ll) <= 64) {
                const int at = atomicAdd(listed, 1);
                if (at < most) list[at] = j * K + k;
            }
        }
        V[i] = v;
    }
}

// The checks of dsfacto_load_csr, predict and evaluate on arrays that are already on the device: row pointers from 0
// to nnz and never falling, column ids rising strictly inside a row and in [0, d), values and labels finite.
// *bad is set if one fails.  A warp takes up to 32 rows at a time (`per`: fewer while that leaves warps without any); once their pointers have been found sound, their entries are
// one stretch that it reads 128 at a time, whatever the rows' lengths.  Columns may fall from one row to the next, so the
// warp counts the places where they do not rise, and the rows that begin at such a place: the two are equal if no row has
// one inside.  Nothing is read outside the arrays whatever they hold.  (One warp per row, 39 M entries: 210 us, most of it
// waiting for one row's pointers and then its entries; now 59 us, 312 MB.)
__global__ void __launch_bounds__(kThreads) validate_rows_kernel(int64_t m, int64_t nnz, int32_t d, const int64_t *__restrict__ indptr,
                                                                 const int32_t *__restrict__ idx, const float *__restrict__ val,
                                                                 const float *__restrict__ y, int *bad, int per) {
    constexpr unsigned FULL = 0xFFFFFFFFu;
    constexpr int U = 4;
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5, warp = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5;
    bool wrong = false;
    for (int64_t i0 = per * warp; i0 < m; i0 += per * nwarps) {
        const int rows = (int)min((int64_t)per, m - i0);
        const int64_t i = i0 + lane;
        int64_t b = 0, e = 0;
        bool sound = true;
        if (lane < rows) {
            b = indptr[i];
            e = indptr[i + 1];
            sound = b >= 0 && b <= e && e <= nnz && (i > 0 || b == 0);
            if (y && !isfinite(y[i])) wrong = true;
        }
        if (!__all_sync(FULL, sound)) { wrong = true; continue; }
        const int64_t from = __shfl_sync(FULL, b, 0), to = __shfl_sync(FULL, e, rows - 1);
        int falls = 0;   // fewer than 2^31 in a lane: it has seen a 32nd of the entries of 32 rows
        for (int64_t t0 = from + lane; t0 < to; t0 += 32 * U) {
            int32_t j[U], before[U];
            float x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t t = t0 + 32 * u;
                j[u] = 0; before[u] = -1; x[u] = 0.f;
                if (t < to) { j[u] = idx[t]; x[u] = val[t]; if (t > from) before[u] = idx[t - 1]; }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (j[u] < 0 || j[u] >= d || !isfinite(x[u])) wrong = true;
                falls += before[u] >= j[u] ? 1 : 0;
            }
        }
        if (b < e && b > from) falls -= idx[b - 1] >= idx[b] ? 1 : 0;
        if (__reduce_add_sync(FULL, falls) != 0) wrong = true;
    }
    if (wrong) *bad = 1;
}

// rows of K floats (caller) <-> rows of Kp floats with zero padding (handle)
__global__ void __launch_bounds__(kThreads) pad_rows_kernel(const float *__restrict__ src, int64_t rows, int K, int Kp, float *__restrict__ dst) {
    const int64_t total = rows * Kp, stride = (int64_t)gridDim.x * kThreads;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < total; i += stride) {
        const int64_t r = i / Kp;
        const int k = (int)(i - r * Kp);
        dst[i] = k < K ? src[r * K + k] : 0.f;
    }
}
__global__ void __launch_bounds__(kThreads) unpad_rows_kernel(const float *__restrict__ src, int64_t rows, int K, int Kp, float *__restrict__ dst) {
    const int64_t total = rows * K, stride = (int64_t)gridDim.x * kThreads;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < total; i += stride) {
        const int64_t r = i / K;
        dst[i] = src[r * Kp + (i - r * K)];
    }
}

}  // namespace dsf
