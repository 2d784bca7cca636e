// lb_limits.cuh -- what the current device has: the dynamic shared-memory limit of kernels whose launches ask
// for differing amounts, and the number of SMs.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

#include "lb_internal.cuh"

namespace lbf {

// Raises the limit of one kernel on the current device to all that a CTA can have, once.  The limit is the
// function's, not the launch's: set per launch or per object to what that one needs, it fails the launches of
// a larger object that another thread, or the same one later, makes.  A repeated set from a concurrent first
// call is harmless, and there is none to make during a capture once an object has been created.
template <auto Kern>
cudaError_t all_shared_memory() {
    static std::atomic<bool> done[MAX_DEVICES];
    int dev = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    cudaFuncAttributes a;
    if ((e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    if ((e = cudaFuncGetAttributes(&a, Kern)) != cudaSuccess) return e;
    e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes);
    if (e == cudaSuccess) done[dev].store(true, std::memory_order_release);
    return e;
}

// SMs of the current device, asked once (1 if it cannot be asked)
inline int device_sms() {
    static std::atomic<int> known[MAX_DEVICES];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return 1;
    n = known[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 1;
        known[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

}  // namespace lbf
