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

// Launches `kernel` so that it may begin before the kernel in front of it on the stream has ended: its CTAs take the SMs as that
// kernel's CTAs leave them, set up their barriers and tensor memory, and wait (ptx::grid_dependency_wait) until the kernel
// has ended and its results are visible.  Every kernel launched this way waits before it touches global memory.
// A kernel that takes tensor memory lets the one behind it begin (ptx::grid_launch_dependents) only once its CTA has it: a CTA of
// that kernel on the same SM might otherwise take it first, then wait for this kernel, and keep it for good.
// A kernel that does not call ptx::grid_launch_dependents lets the kernel behind begin as its own CTAs end, and still saves most of
// the gap.  So do the row kernels of more than 8192 columns: several of their CTAs fit an SM, so those of the kernel behind would
// begin beside the ones that work and lie unevenly when their turn comes, and each has a fixed share of the rows.  us per call, calling it at
// the begin -> not at all (without overlap): two-read bfloat16 3937 x 43008 217 -> 186 (189), float32 5081 x 40632 317 -> 296 (298), bfloat16
// 60 x 36864 12.4 -> 6.2 (8.2); cluster bfloat16 300 x 44000 21.1 -> 17.3 (19.3); shared memory bfloat16 500 x 30000 24.5 -> 22.1 (24.7).
// Back to back, small calls took 2 us more each: 4096 x 1000 float32 row Softmax 6.2 -> 4.6 us, attention of 2 x 128 8.2 -> 5.4,
// projection of 64 rows 8.2 -> 5.3, weights of one head of 256 8.4 -> 6.5.
// `cluster` CTAs form a cluster; `cooperative`: the whole grid is resident at once, or the launch fails.
template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                                     int cluster, bool cooperative, Args... args) {
    cudaLaunchAttribute attr[3];
    unsigned n = 0;
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = static_cast<unsigned>(cluster);
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    if (cooperative) {
        attr[n].id = cudaLaunchAttributeCooperative;
        attr[n++].val.cooperative = 1;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

}  // namespace attnw
