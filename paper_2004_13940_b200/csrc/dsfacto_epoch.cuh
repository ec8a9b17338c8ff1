// What the kernels of an epoch share: scalars on the device, the report to the host, overlapped launches.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace dsf {

// Scalars of an epoch that stay on the device between its kernels.
struct EpochState {
    double loss, g, w2, v2;        // of the last recompute pass
    float w0;
    unsigned done;                 // CTAs of the recompute pass that have delivered their sums
    int err[3];                    // bounds-checked build: code and value of the first failed check
    int bad;                       // caller data on the device has failed a check (zero between calls)
    uint32_t epochs;               // reports of epochs (and other recompute passes) so far
    unsigned long long t0, t1;     // device clock: start of the update loop, start of the recompute pass
    unsigned long long ns[2];      // update loop, recompute pass: sums over the segments of an epoch
};
// What kernels tell the host, in mapped host memory: words of 64 bits, the number of the report in the upper half and 32 bits
// of its contents in the lower.  Each word arrives whole and says by itself whether it has arrived, so the kernel neither waits
// for its writes to have crossed the link before it writes a last one (1.8 us for the round trip of a fence) nor writes them in
// any order; the host has the report when all its words carry the number.
struct EpochBody {                 // end of an epoch, or of a recompute pass
    double loss, g, w2, v2;
    unsigned long long ns[2];
    float w0;
    int err[3];
};
struct CallBody {                  // end of a scoring or copying kernel
    double loss, g;
    int bad, unused;
};
template <class Body>
constexpr int kReportWords = (int)(sizeof(Body) / sizeof(uint32_t));
static_assert(sizeof(EpochBody) % 4 == 0 && kReportWords<EpochBody> <= 32 && sizeof(CallBody) % 4 == 0 && kReportWords<CallBody> <= 32, "a word per lane");
struct Report {
    unsigned long long epoch[kReportWords<EpochBody>], call[kReportWords<CallBody>];
    int bad;                       // caller data on the device has failed a check (read after a wait for the stream)
};
__device__ __forceinline__ void store_report_word(unsigned long long *word, uint32_t number, uint32_t contents) {
    asm volatile("st.relaxed.sys.global.u64 [%0], %1;" ::"l"(word), "l"((unsigned long long)number << 32 | contents) : "memory");
}
// by a warp, from shared memory
template <class Body>
__device__ __forceinline__ void store_report(unsigned long long *words, uint32_t number, const Body &body) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    if (lane < kReportWords<Body>) store_report_word(words + lane, number, reinterpret_cast<const uint32_t *>(&body)[lane]);
}

__device__ __forceinline__ unsigned long long device_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Kernels of an epoch are launched with programmatic stream serialisation: the next one may start its prologue
// early and waits here for everything before it (no-op for an ordinary launch).
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace dsf
