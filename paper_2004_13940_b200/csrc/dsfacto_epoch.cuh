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
    unsigned long long epochs;     // reports of epochs (and other recompute passes) so far
    unsigned long long t0, t1;     // device clock: start of the update loop, start of the recompute pass
    unsigned long long ns[2];      // update loop, recompute pass: sums over the segments of an epoch
};
// What the host waits for at the end of an epoch (mapped host memory).
struct EpochReport {
    double loss, g, w2, v2;
    float w0;
    int err[3];
    int bad;
    unsigned long long ns[2];
    unsigned long long seq, epochs;   // last number reported by scoring and copying kernels; by recompute passes
};

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
