// dsfacto_score_loss_noalloc: scores, loss sum and multiplier sum of a batch of rows, for callers that
// must not allocate.
//
// Who needs this: code that runs where device allocation is forbidden or unsafe - inside a region
// that another framework has closed to cudaMalloc (a memory pool that owns the whole device, a
// serving loop with a fixed memory budget), or from a thread that must never block on the
// driver's allocation lock.  Such a caller already owns device buffers with the rows, the
// parameters and room for the results; the only thing the ordinary path would still allocate is the
// per-CTA partial sums of the loss reduction.  Here those live in a fixed array that is part of
// the library image.
#include "dsfacto.h"
#include "dsfacto_common.cuh"
#include "dsfacto_recompute.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>

namespace {

using namespace dsf;

constexpr int64_t kMaxRows = (int64_t)1 << 26;   // most rows of a call
constexpr int kMaxCtas = 32768;      // CTAs whose partial sums fit the scratch array
constexpr int kMaxDevices = 64;

// Scratch of the reduction: four sums per CTA (two of them in use), 1 MiB, and the number of CTAs that have delivered
// theirs, which every launch leaves at zero.  Every GPU that
// loads the library holds one copy until the process exits.  Each call overwrites the slots it
// uses before it reads them, so nothing has to start at zero; the contents of the last call stay.
static __device__ __align__(256) double g_noalloc_partials[4 * kMaxCtas];
static __device__ unsigned g_noalloc_done;

// their device addresses per device (the symbols themselves are only host-side stand-ins); every writer stores the
// same value, and the second is stored before the first is published
std::atomic<double *> g_partials_addr[kMaxDevices];
std::atomic<unsigned *> g_done_addr[kMaxDevices];

// The recompute kernel of the epoch (eq. (fm_model2), the multiplier G, the loss) without its stores of the
// auxiliaries and without per-column pairs, for which there is no room: w_j and sum_k v_jk^2 come from w and V.
template <int LG, int NV>
void launch_score_loss(const RefreshArgs &a, int32_t d, cudaStream_t st) {
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t rows = RefreshCfg<LG, NV>::ROWS;
    const int64_t grid = std::min<int64_t>((a.n + rows - 1) / rows, (int64_t)sms * RefreshCfg<LG, NV>::CTAS);
    const unsigned ctas = (unsigned)std::min<int64_t>(grid, kMaxCtas);
    // Whether nothing is requested behind the end of a row (TRIM), or its last entry again.  Not requesting saves look-ups and
    // data where the rows that a warp takes side by side differ in length, and costs a look at every entry.  12 M entries over
    // 50 to 1 M columns, rows of 39, 20 to 60, 1 to 77 and 1 to 12 entries, columns drawn evenly and by a power law: the time
    // that repeating takes, over the time without, is 0.96 to 1.20 for 32-byte rows, 0.98 to 1.22 for 64-byte, 0.99 to 1.13 for
    // 128-byte and 1.00 to 1.09 for 512-byte rows.  256-byte rows: 0.97 to 1.00 over tables of up to 150 KB, which an L1 holds
    // whole, 0.98 to 1.03 over 175 to 225 KB, 0.99 to 1.27 over larger ones.  Two widths are better off repeating more often
    // than not: 16-byte rows (0.86 to 1.11, below 1 in 16 of 24 cases) and 1-KB rows over up to 320 KB (0.96 to 1.12, in 21 of 32).
    constexpr bool repeats = (LG == 1 && NV == 1) || (LG == 8 && NV == 8), by_table = LG == 8 && NV == 2;
    if constexpr (!repeats) {
        if (!by_table || (int64_t)d * 4 * LG * NV * (int64_t)sizeof(float) > ((int64_t)192 << 10)) {
            refresh_kernel<LG, NV, kScoreSums, true, true><<<ctas, kThreads, 0, st>>>(a);
            return;
        }
    }
    if constexpr (repeats || by_table) refresh_kernel<LG, NV, kScoreSums, true, false><<<ctas, kThreads, 0, st>>>(a);
}

}  // namespace

extern "C" int dsfacto_score_loss_noalloc(int64_t m, int32_t d, int32_t K, int32_t loss, const int64_t *indptr_dev,
                                          const int32_t *indices_dev, const float *values_dev, const float *y_dev,
                                          float w0, const float *w_dev, const float *V_dev, float *scores_dev,
                                          double *sums_dev, void *cuda_stream) {
    if (m < 1 || d < 1 || !indptr_dev || !indices_dev || !values_dev || !y_dev || !w_dev || !V_dev || !scores_dev || !sums_dev)
        return DSFACTO_ERR_INVALID_ARG;
    // rows of V are read 16 bytes at a time: a pointer that is not 16-byte aligned would fault on the device,
    // so it is refused here instead
    if ((reinterpret_cast<uintptr_t>(V_dev) & 15u) != 0) return DSFACTO_ERR_INVALID_ARG;
    if (loss != DSFACTO_SQUARED && loss != DSFACTO_LOGISTIC) return DSFACTO_ERR_INVALID_ARG;
    if (!std::isfinite(w0)) return DSFACTO_ERR_INVALID_ARG;
    // rows of V are read as float4 lane groups: K must be 4, 8, 16, 32, 64, 128 or 256
    if (K < 4 || K > 256 || (K & (K - 1)) != 0) return DSFACTO_ERR_INVALID_ARG;
    if (m > kMaxRows) return DSFACTO_ERR_INVALID_ARG;

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return DSFACTO_ERR_CUDA;
    if (!g_partials_addr[dev]) {  // first call on this device: resolve the array's device address
        double *p = nullptr;
        if (cudaGetSymbolAddress((void **)&p, g_noalloc_partials) != cudaSuccess || !p) return DSFACTO_ERR_CUDA;
        unsigned *q = nullptr;
        if (cudaGetSymbolAddress((void **)&q, g_noalloc_done) != cudaSuccess || !q) return DSFACTO_ERR_CUDA;
        g_done_addr[dev] = q;
        g_partials_addr[dev] = p;
    }
    RefreshArgs a{};
    a.n = m; a.indptr = indptr_dev; a.idx = indices_dev; a.val = values_dev; a.y = y_dev; a.w = w_dev; a.V = V_dev; a.w0 = w0;
    a.loss = loss; a.f_out = scores_dev; a.sums_out = sums_dev; a.partials = g_partials_addr[dev]; a.done = g_done_addr[dev];
    cudaStream_t st = (cudaStream_t)cuda_stream;
    switch (K) {
    case 4: launch_score_loss<1, 1>(a, d, st); break;
    case 8: launch_score_loss<2, 1>(a, d, st); break;
    case 16: launch_score_loss<4, 1>(a, d, st); break;
    case 32: launch_score_loss<8, 1>(a, d, st); break;
    case 64: launch_score_loss<8, 2>(a, d, st); break;
    case 128: if (wide_recompute_groups(d, K)) launch_score_loss<16, 2>(a, d, st); else launch_score_loss<8, 4>(a, d, st); break;
    case 256: if (wide_recompute_groups(d, K)) launch_score_loss<16, 4>(a, d, st); else launch_score_loss<8, 8>(a, d, st); break;
    default: return DSFACTO_ERR_INVALID_ARG;
    }
    if (cudaGetLastError() != cudaSuccess) return DSFACTO_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return DSFACTO_ERR_CUDA;
    return DSFACTO_OK;
}
