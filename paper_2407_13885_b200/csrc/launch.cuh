// Host-side launch helper shared by the kernels' launchers.
#pragma once
#include <atomic>

#include <cuda_runtime.h>

namespace attnw {

constexpr int kMaxDevices = 64;

// Lets `Kernel` use `bytes` of dynamic shared memory on the current device and, with `large_clusters`, clusters of more
// than 8 CTAs.  The setting belongs to the (kernel, device) pair and stays, so the driver is asked once per pair and not
// on every call; every instantiation has one flag per device (and internal linkage: two builds of the library in one
// process have kernels of their own).  `bytes` is the most that any launch of the kernel asks for.
template <auto Kernel>
static inline cudaError_t allow_smem(int bytes, bool large_clusters = false) {
    static std::atomic<unsigned long long> done{0};
    static_assert(kMaxDevices <= 64, "one bit per device");
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (done.load(std::memory_order_relaxed) >> dev & 1) return cudaSuccess;
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && large_clusters) e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) done.fetch_or(1ull << dev, std::memory_order_relaxed);
    return e;
}

}  // namespace attnw
