// Shared device helpers of the DS-FACTO kernels (sm_100a).
//
// Factor-row layout used by every kernel: a row (v_j or a_i) occupies Kp = 4*LG*NV floats, 16-byte
// aligned, K <= Kp, padding kept at zero.  A "lane group" of LG consecutive lanes (LG a power of
// two <= 32) owns one row: lane l holds float4 number l, l+LG, ... (NV of them), so the group's
// loads of one row are coalesced.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace dsf {

constexpr int kThreads = 256;
constexpr uint32_t kNoCol = 0xFFFFFFFFu;

template <int LG>
__device__ __forceinline__ uint32_t group_mask() {
    if (LG == 32) return 0xFFFFFFFFu;
    const uint32_t lane = threadIdx.x & 31u;
    return ((1u << LG) - 1u) << (lane & ~uint32_t(LG - 1));
}

// acc += c * r on four floats with two packed fp32x2 multiply-adds (each half rounds exactly as a scalar fmaf).
// (512-byte rows in the tile sweep: 21.3 -> 19.4 ms per sweep of 400 M entries; 64-byte rows: no change.)
__device__ __forceinline__ void fma4(float4 &acc, const float c, const float4 r) {
    const float2 cc = make_float2(c, c);
    const float2 lo = __ffma2_rn(make_float2(r.x, r.y), cc, make_float2(acc.x, acc.y));
    const float2 hi = __ffma2_rn(make_float2(r.z, r.w), cc, make_float2(acc.z, acc.w));
    acc = make_float4(lo.x, lo.y, hi.x, hi.y);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// deterministic CTA-wide sum of two doubles; result valid in thread 0
__device__ __forceinline__ void block_sum2(double &a, double &b) {
    __shared__ double sh[2][kThreads / 32];
    a = warp_sum(a);
    b = warp_sum(b);
    const int wid = threadIdx.x >> 5, ln = threadIdx.x & 31;
    if (ln == 0) { sh[0][wid] = a; sh[1][wid] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double x = 0.0, y = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) { x += sh[0][i]; y += sh[1][i]; }
        a = x; b = y;
    }
}

// the same for four.  Lanes hand half of their sums over while they halve: after two steps a lane adds up one of the four, so
// a warp shuffles six doubles instead of twenty, and one warp adds up what the warps have left (the chain of 8 x 4 additions
// by thread 0 and the longer shuffles were part of the end of a recompute pass, which does this twice at its end: 650 k entries 10.3 -> 10.0 us, call to call 28.4 -> 28.0; 20 k entries 19.1 -> 17.5).
__device__ __forceinline__ double half_sum(double (&s)[2], bool upper, int o) {
    return (upper ? s[1] : s[0]) + __shfl_xor_sync(0xFFFFFFFFu, upper ? s[0] : s[1], o);
}
__device__ __forceinline__ void block_sum4(double (&s)[4]) {
    __shared__ double sh[4 * (kThreads / 32)];
    static_assert(kThreads / 32 == 8, "a double per lane of one warp");
    const int wid = threadIdx.x >> 5, ln = threadIdx.x & 31;
    double lo[2] = {s[0], s[1]}, hi[2] = {s[2], s[3]};
    double two[2] = {half_sum(lo, (ln & 1) != 0, 1), half_sum(hi, (ln & 1) != 0, 1)};   // sums (ln & 1) and 2 + (ln & 1)
    double x = half_sum(two, (ln & 2) != 0, 2);                                         // sum (ln & 3)
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    __syncthreads();   // (an earlier call's reads)
    if (ln < 4) sh[4 * wid + ln] = x;
    __syncthreads();
    if (wid == 0) {
        x = sh[ln];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] = __shfl_sync(0xFFFFFFFFu, x, c);
    }
}

}  // namespace dsf
