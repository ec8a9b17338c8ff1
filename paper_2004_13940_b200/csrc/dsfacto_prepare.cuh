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
// *bad is set if one fails.  One warp per row; nothing is read outside the arrays whatever they hold.
__global__ void __launch_bounds__(kThreads) validate_rows_kernel(int64_t m, int64_t nnz, int32_t d, const int64_t *__restrict__ indptr,
                                                                 const int32_t *__restrict__ idx, const float *__restrict__ val,
                                                                 const float *__restrict__ y, int *bad) {
    const int lane = (int)(threadIdx.x & 31u);
    const int64_t nwarps = ((int64_t)gridDim.x * kThreads) >> 5;
    bool wrong = false;
    for (int64_t i = ((int64_t)blockIdx.x * kThreads + threadIdx.x) >> 5; i < m; i += nwarps) {
        const int64_t b = indptr[i], e = indptr[i + 1];
        if (b < 0 || e < b || e > nnz || (i == 0 && b != 0)) { wrong = true; continue; }
        if (y && !isfinite(y[i])) wrong = true;
        for (int64_t t = b + lane; t < e; t += 32) {
            const int32_t j = idx[t];
            if (j < 0 || j >= d || !isfinite(val[t]) || (t > b && idx[t - 1] >= j)) wrong = true;
        }
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
