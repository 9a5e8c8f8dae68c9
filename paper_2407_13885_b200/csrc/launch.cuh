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

// Launches `kernel` so that it may begin as soon as every CTA of the kernel in front on the stream has ended: what lies between the
// end of one kernel and the begin of the next runs beside its set-up, and it waits (ptx::grid_dependency_wait) until the results in
// front are visible.  Every kernel launched this way waits before it touches global memory.  Back to back, small calls took about 2 us
// more each: 4096 x 1000 float32 row Softmax 6.2 -> 4.6 us, attention of 2 x 128 8.2 -> 5.9, projection of 64 rows 6.2 -> 4.3, weights
// of one head of 256 8.6 -> 7.2.
// No kernel lets the one behind begin earlier (griddepcontrol.launch_dependents).  Its CTAs would take room as CTAs of the kernel in front
// leave it, not evenly, where each has a fixed share of the work, and clusters would not all find their SMs.  us, two calls one behind the
// other, early / as now / without overlap: rows 1000 x 131072 behind weights of 24 x 1000 236 / 157 / 162, rows 600 x 44000 behind 9 x 256
// 55.9 / 39.7 / 43.9, weights of 82 x 752 behind themselves 46.3 / 30.3 / 32.7.  It saved another 0.3 to 0.5 us between the smallest
// calls of the tensor-core kernels (one head of 256 7.2 -> 6.8), and it has to come after a CTA has its tensor memory: a CTA of the
// kernel behind on the same SM might otherwise take that first, then wait for this kernel, and keep it for good.
// `cluster` CTAs form a cluster.
template <typename... Params, typename... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                                     int cluster, Args... args) {
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = static_cast<unsigned>(cluster);
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
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
