// C ABI of libattnw.so: argument validation, tensor-map encoding and kernel launches.
// The contract of every entry point is stated in include/attnw.h.
#include <atomic>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <type_traits>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/attnw.h"
#include "launch.cuh"
#include "attnw_fused.cuh"
#include "attn_fused.cuh"
#include "attn_onepass.cuh"
#include "project_qk.cuh"
#include "attnw_resident.cuh"
#include "attnw_gridrow.cuh"
#include "softmax_rows.cuh"
#include "softmax_rows_smem.cuh"

namespace {

using namespace attnw;

constexpr int kMaxGridrowAreas = 8;  // exchange areas of the grid-row kernel per device
constexpr uint32_t kSiteSelfTest = 127;  // wait site of attnw_selftest_wait_timeout (low byte of the status word)

// Not part of any product path: one thread waits, with the caller's limit, on an mbarrier that nobody arrives on,
// gives up, records the site in the per-device status word and returns - the unwinding every kernel's bounded wait
// follows, made reachable for a test without touching the waits of the real kernels.
__global__ void wait_timeout_selftest_kernel(long long limit_cycles) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bar, 1);
        ptx::mbar_fence_init();
        const long long t0 = clock64();
        while (!ptx::mbar_try_wait(&bar, 0u)) {
            if (clock64() - t0 > limit_cycles) {
                atomicCAS(&g_attnw_status, 0u, 0x80000000u | kSiteSelfTest);
                break;
            }
        }
    }
}

// Reads the current device's status word after the caller has synchronised; a recorded failure is cleared and
// reported once.
int read_and_clear_status(unsigned int* word_out) {
    unsigned int word = 0;
    if (cudaMemcpyFromSymbol(&word, attnw::g_attnw_status, sizeof(word)) != cudaSuccess) return ATTNW_ERR_CUDA;
    if (word_out) *word_out = word;
    if (word == 0) return ATTNW_OK;
    const unsigned int zero = 0;
    if (cudaMemcpyToSymbol(attnw::g_attnw_status, &zero, sizeof(zero)) != cudaSuccess) return ATTNW_ERR_CUDA;
    return ATTNW_ERR_TIMEOUT;
}
constexpr int kVersion = 100;  // 0.1.0

std::atomic<long long> g_launches{0};
std::atomic<int> g_rows_variant{0};   // 0 = tier by row length, 1 = caching (register tier only), 2 = recomputing with a second read, 3 = recomputing from registers
std::atomic<int> g_attn_variant{0};   // 0 = default (one pass), 1 = two-pass, 2 = one pass
std::atomic<int> g_fused_variant{0};  // 0 = choose by shape, 1 = two-pass, 2 = SRAM-resident, 3 = SRAM-resident, owner-reduce exchange
constexpr double kTwoPassPerSm = 0.9;  // measured: per-SM throughput of the two-pass kernel relative to the resident one
std::mutex g_mutex;

struct DeviceInfo {
    std::atomic<bool> ready{false};  // cc_major and sm_count are valid
    int cc_major = 0;
    int sm_count = 0;
    int fused_pairs[2][2] = {};  // [d == 128][float32 P]: co-resident two-CTA clusters of the two-pass kernel, 0 = not asked yet
    int resident_clusters[2][kMaxClusterCtas + 1] = {};  // [d == 128][cluster size]: co-resident clusters, 0 = not asked yet
    // fork/join objects for launches that split a call over two kernels (created on first use)
    cudaStream_t side_stream = nullptr;
    cudaEvent_t fork_event = nullptr, join_event = nullptr;
    std::atomic<int> gridrow_clusters[2][2][17] = {};  // resident clusters of 2..16 CTAs of the grid-row kernel, [d == 128][P is float32][CTAs], 0 = not asked yet
    std::atomic<int> attn_clusters[2][5] = {};  // resident clusters of 2 and 4 CTAs of the one-pass attention kernel, [d == 128][CTAs]
    int rc_clusters[2][17] = {};  // resident clusters of 1..16 CTAs of the register-cluster row kernel, [P is float32][CTAs]
};
std::mutex g_split_mutex;
DeviceInfo g_devices[kMaxDevices];

// Exchange areas of the grid-row kernel.  A launch owns its area until it ends; launches on one stream follow each other,
// so a stream keeps the area it has, and a program with one stream uses one.  A stream that has none takes a new one, up
// to kMaxGridrowAreas per device, or one whose last launch is known to have ended, or else waits for the area that was
// given to its stream first.  Stream ids are never used twice, unlike stream handles.
struct GridrowArea {
    uint4* xchg = nullptr;
    unsigned long long stream_id = 0;
    uint32_t tag = 0;           // the next unused message tag
    cudaEvent_t last = nullptr; // the end of the last launch ...
    bool recorded = false;      // ... if it was recorded: not while the device has had one stream only
};
struct GridrowAreas {
    std::mutex mutex;  // held over the launch, so that no other stream takes the area before its event is recorded
    GridrowArea area[kMaxGridrowAreas];
    int count = 0, next_victim = 0;
    bool several_streams = false;
};
GridrowAreas g_gridrow_areas[kMaxDevices];

// The tags *base + 1 ... *base + n of an exchange area's messages for one launch, from the counter `next`; 0 is never a tag.
// true: the tags had run out (after about 2e9 row blocks) and start over, so the area must be cleared in front of the launch.  Where
// a message lies depends on the launch's groups: messages of other shapes may have stood there since the low tags were last in use.
// The upper half of the tags belongs to launches of attnw_fused_noalloc in graphs, which repeat them on every replay.
constexpr uint32_t kLastTag = 0x7fffffffu, kCapturedTagBase = kLastTag;
bool take_tags(uint32_t* next, uint32_t n, uint32_t* base) {
    const bool start_over = n > kLastTag - *next;
    if (start_over) *next = 0;
    *base = *next;
    *next += n;
    return start_over;
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
std::atomic<EncodeTiledFn> g_encode_tiled{nullptr};

// Current device's cached properties; returns an attnw_status.
int current_device(DeviceInfo** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    DeviceInfo& d = g_devices[dev];
    if (!d.ready.load(std::memory_order_acquire)) {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (cudaDeviceGetAttribute(&d.cc_major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            (void)cudaGetLastError();
            return ATTNW_ERR_CUDA;
        }
        d.ready.store(true, std::memory_order_release);
    }
    *out = &d;
    return d.cc_major == 10 ? ATTNW_OK : ATTNW_ERR_UNSUPPORTED;
}

int load_encoder() {
    if (g_encode_tiled.load(std::memory_order_relaxed)) return ATTNW_OK;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || fn == nullptr) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    g_encode_tiled.store(reinterpret_cast<EncodeTiledFn>(fn), std::memory_order_relaxed);
    return ATTNW_OK;
}

// Row-major [dim2][dim1][dim0] tensor, box {box0, box1, 1}, 128-byte swizzle (box0 * esize == 128).
int encode_3d(CUtensorMap* map, CUtensorMapDataType dtype, size_t esize, const void* base, uint64_t dim0,
              uint64_t dim1, uint64_t dim2, uint32_t box0, uint32_t box1) {
    const cuuint64_t dims[3] = {dim0, dim1, dim2};
    const cuuint64_t strides[2] = {dim0 * esize, dim0 * dim1 * esize};
    const cuuint32_t box[3] = {box0, box1, 1};
    const cuuint32_t elem_strides[3] = {1, 1, 1};
    CUresult r = g_encode_tiled.load(std::memory_order_relaxed)(map, dtype, 3, const_cast<void*>(base), dims, strides, box, elem_strides,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? ATTNW_OK : ATTNW_ERR_CUDA;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool overlaps(const void* a, unsigned long long a_bytes, const void* b, unsigned long long b_bytes) {
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(a), b0 = reinterpret_cast<uintptr_t>(b);
    return a0 < b0 + b_bytes && b0 < a0 + a_bytes;
}

// Host-only checks of the fused call; no CUDA call is made here.
int validate_fused(const void* Q, const void* K, const void* P, int B, int H, int N, int d, float scale,
                   size_t p_esize) {
    if (!Q || !K || !P) return ATTNW_ERR_NULL_POINTER;
    if (B < 1 || H < 1 || N < 1 || d < 1) return ATTNW_ERR_BAD_SHAPE;
    if (!(scale >= 0.0f) || !std::isfinite(scale)) return ATTNW_ERR_BAD_SHAPE;
    const long long bh = static_cast<long long>(B) * H;
    if (bh > INT_MAX) return ATTNW_ERR_BAD_SHAPE;
    const long long ctas = bh * ((static_cast<long long>(N) + kRowsPerCta - 1) / kRowsPerCta);
    if (ctas > INT_MAX) return ATTNW_ERR_BAD_SHAPE;
    if (N > (1 << 24)) return ATTNW_ERR_BAD_SHAPE;  // keeps every tensor-map stride below 2^40 bytes
    if (d != 64 && d != 128) return ATTNW_ERR_UNSUPPORTED;
    if (!aligned16(Q) || !aligned16(K) || !aligned16(P)) return ATTNW_ERR_MISALIGNED;
    if ((static_cast<unsigned long long>(N) * p_esize) % 16 != 0) return ATTNW_ERR_MISALIGNED;
    if (static_cast<unsigned long long>(N) * N * p_esize >= (1ull << 40)) return ATTNW_ERR_BAD_SHAPE;
    const unsigned long long qk_bytes = static_cast<unsigned long long>(bh) * N * d * 2ull;
    const unsigned long long p_bytes = static_cast<unsigned long long>(bh) * N * N * p_esize;
    if (overlaps(P, p_bytes, Q, qk_bytes) || overlaps(P, p_bytes, K, qk_bytes)) return ATTNW_ERR_ALIASING;
    return ATTNW_OK;
}

template <int D, typename OutT>
int launch_fused(DeviceInfo* dev, const void* Q, const void* K, void* P, int BH, int N, float scale,
                 cudaStream_t stream, bool allow_key_split = true) {
    using L = FusedSmem<D>;
    auto kernel = attnw_fused_kernel<D, OutT>;
    CUtensorMap tm_q, tm_k, tm_p;
    int rc = encode_3d(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Q, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) {
        if (sizeof(OutT) == 2)
            rc = encode_3d(&tm_p, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, P, N, N, BH, 64, kTile);
        else
            rc = encode_3d(&tm_p, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, P, N, N, BH, 32, kTile);
    }
    if (rc != ATTNW_OK) return rc;
    if (allow_smem<attnw_fused_kernel<D, OutT>>(L::kDynamicBytes) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    const int row_blocks = (N + kRowsPerCta - 1) / kRowsPerCta;
    const float scale_log2e = static_cast<float>(static_cast<double>(scale) * 1.4426950408889634074);
    const long long ctas = static_cast<long long>(BH) * row_blocks;
    // Two CTAs per 256-row block (each walks half of the key tiles; see the kernel) when that fills the device
    // better: CTAs of half the length in waves of `pairs` clusters against whole CTAs in waves of `sm_count`
    // (N = 16384, B*H = 8: 512 CTAs = 4 waves of 148 become 7 half-length waves of 74 pairs; a call with fewer
    // CTAs than SMs simply finishes in half the time).
    int key_split = 1;
    if (allow_key_split && ((N + kTile - 1) / kTile) % 2 == 0 && 2 * ctas <= INT_MAX) {
        int& pairs = dev->fused_pairs[D == 128 ? 1 : 0][sizeof(OutT) == 2 ? 0 : 1];
        if (pairs == 0) {
            cudaLaunchAttribute a[1];
            a[0].id = cudaLaunchAttributeClusterDimension;
            a[0].val.clusterDim.x = 2;
            a[0].val.clusterDim.y = 1;
            a[0].val.clusterDim.z = 1;
            cudaLaunchConfig_t c = {};
            c.blockDim = dim3(kFusedThreads, 1, 1);
            c.gridDim = dim3(static_cast<unsigned>(2 * dev->sm_count), 1, 1);
            c.dynamicSmemBytes = L::kDynamicBytes;
            c.attrs = a;
            c.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kernel, &c) != cudaSuccess || n < 1) {
                (void)cudaGetLastError();
                n = -1;
            }
            pairs = n;
        }
        if (pairs > 0) {
            const long long whole_waves = (ctas + dev->sm_count - 1) / dev->sm_count;
            const long long half_waves = (ctas + pairs - 1) / pairs;
            if (half_waves * 51 < whole_waves * 100) key_split = 2;  // 2 % for the exchange
        }
    }
    if (key_split == 1) {
        kernel<<<static_cast<unsigned>(ctas), kFusedThreads, L::kDynamicBytes, stream>>>(tm_q, tm_k, tm_p, N, row_blocks,
                                                                                         scale_log2e, 1);
    } else {
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = 2;
        a[0].val.clusterDim.y = 1;
        a[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t c = {};
        c.blockDim = dim3(kFusedThreads, 1, 1);
        c.gridDim = dim3(static_cast<unsigned>(2 * ctas), 1, 1);
        c.dynamicSmemBytes = L::kDynamicBytes;
        c.stream = stream;
        c.attrs = a;
        c.numAttrs = 1;
        if (cudaLaunchKernelEx(&c, kernel, tm_q, tm_k, tm_p, N, row_blocks, scale_log2e, 2) != cudaSuccess) {
            (void)cudaGetLastError();
            return ATTNW_ERR_CUDA;
        }
    }
    if (cudaGetLastError() != cudaSuccess) return ATTNW_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ATTNW_OK;
}

// How many clusters of `cluster_ctas` CTAs of the resident kernel the device can hold at once (cached).
template <int D, int CMAX>
int resident_max_clusters_impl(DeviceInfo* dev, int cluster_ctas) {  // (both exchange forms have the same footprint)
    int& cached = dev->resident_clusters[D == 128 ? 1 : 0][cluster_ctas];
    if (cached != 0) return cached;
    using L = ResidentSmem<D, CMAX>;
    auto kernel = attnw_resident_kernel<D, CMAX, false>;
    if (allow_smem<attnw_resident_kernel<D, CMAX, false>>(L::kDynamicBytes, CMAX > 8) != cudaSuccess) {
        (void)cudaGetLastError();
        return cached = -1;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cluster_ctas);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kResidentThreads, 1, 1);
    cfg.dynamicSmemBytes = L::kDynamicBytes;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(cluster_ctas * dev->sm_count), 1, 1);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        n = -1;
    }
    return cached = n;
}

template <int D>
int resident_max_clusters(DeviceInfo* dev, int cluster_ctas) {
    return cluster_ctas <= 8 ? resident_max_clusters_impl<D, 8>(dev, cluster_ctas)
                             : resident_max_clusters_impl<D, 16>(dev, cluster_ctas);
}

// SRAM-resident single-pass kernel: one cluster of ceil(N / 512) CTAs per 128-row block, persistent over
// a list of row blocks.  Returns ATTNW_ERR_UNSUPPORTED when the device cannot co-schedule such a cluster.
template <int D, int CMAX, bool OWNER>
int launch_resident_impl(DeviceInfo* dev, const void* Q, const void* K, void* P, int BH, int N, float scale,
                         cudaStream_t stream) {
    using L = ResidentSmem<D, CMAX>;
    auto kernel = attnw_resident_kernel<D, CMAX, OWNER>;
    CUtensorMap tm_q, tm_k, tm_p;
    int rc = encode_3d(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Q, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_p, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, P, N, N, BH, 64, kTile);
    if (rc != ATTNW_OK) return rc;
    if (allow_smem<attnw_resident_kernel<D, CMAX, OWNER>>(L::kDynamicBytes, CMAX > 8) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    const int cluster_ctas = (N + kSlab - 1) / kSlab;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cluster_ctas);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kResidentThreads, 1, 1);
    cfg.dynamicSmemBytes = L::kDynamicBytes;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int max_clusters = resident_max_clusters<D>(dev, cluster_ctas);
    if (max_clusters < 1) return ATTNW_ERR_UNSUPPORTED;
    const int row_blocks = (N + kTile - 1) / kTile;
    const long long total_items = static_cast<long long>(BH) * row_blocks;
    if (total_items > INT_MAX) return ATTNW_ERR_BAD_SHAPE;
    const int clusters = total_items < max_clusters ? static_cast<int>(total_items) : max_clusters;
    cfg.gridDim = dim3(static_cast<unsigned>(clusters * cluster_ctas), 1, 1);
    const float scale_log2e = static_cast<float>(static_cast<double>(scale) * 1.4426950408889634074);
    if (cudaLaunchKernelEx(&cfg, kernel, tm_q, tm_k, tm_p, N, static_cast<int>(total_items), cluster_ctas, scale_log2e) !=
        cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ATTNW_OK;
}

template <int D>
int launch_resident(DeviceInfo* dev, const void* Q, const void* K, void* P, int BH, int N, float scale,
                    cudaStream_t stream, bool owner_reduce = false) {
    const bool small = (N + kSlab - 1) / kSlab <= 8;
    if (owner_reduce)
        return small ? launch_resident_impl<D, 8, true>(dev, Q, K, P, BH, N, scale, stream)
                     : launch_resident_impl<D, 16, true>(dev, Q, K, P, BH, N, scale, stream);
    return small ? launch_resident_impl<D, 8, false>(dev, Q, K, P, BH, N, scale, stream)
                 : launch_resident_impl<D, 16, false>(dev, Q, K, P, BH, N, scale, stream);
}

// The geometry of a grid-row launch: groups of ceil(N / 256) CTAs, as many as fit one CTA per SM and have work.
struct GridrowShape {
    int group_ctas, n_groups, total_items;
    bool clusters;     // each group is a cluster (else: the grid is cooperative)
    uint32_t longest;  // row blocks of the longest list = message tags the launch uses
};
// How many clusters of `ctas` CTAs of the grid-row kernel the device holds at once; -1 = none.
template <int D, typename OutT>
int gridrow_max_clusters(DeviceInfo* dev, int ctas) {
    std::atomic<int>& memo = dev->gridrow_clusters[D == 128][sizeof(OutT) == 4][ctas];
    int n = memo.load(std::memory_order_relaxed);
    if (n != 0) return n;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(ctas);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(gr::kThreads, 1, 1);
    cfg.gridDim = dim3(static_cast<unsigned>(ctas * dev->sm_count), 1, 1);
    cfg.dynamicSmemBytes = gr::Smem<D>::kDynamicBytes;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, gr::attnw_gridrow_kernel<D, OutT>, &cfg) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        n = -1;
    }
    memo.store(n, std::memory_order_relaxed);
    return n;
}

// Returns ATTNW_ERR_UNSUPPORTED when `max_ctas` cannot hold a whole group.
template <int D, typename OutT>
int gridrow_shape(DeviceInfo* dev, int BH, int N, int max_ctas, GridrowShape* out) {
    const long long total = static_cast<long long>(BH) * ((N + kTile - 1) / kTile);
    if (total > INT_MAX) return ATTNW_ERR_BAD_SHAPE;
    const int C = (N + gr::kSlabCols - 1) / gr::kSlabCols;
    if (C > max_ctas || C > gr::kMaxGroupCtas) return ATTNW_ERR_UNSUPPORTED;
    if (allow_smem<gr::attnw_gridrow_kernel<D, OutT>>(gr::Smem<D>::kDynamicBytes, true) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    out->group_ctas = C;
    out->total_items = static_cast<int>(total);
    out->n_groups = max_ctas / C;
    auto rounds = [&](int groups) { return (total + groups - 1) / groups; };
    // The CTAs of a group wait for one another, so they must be resident together: as a cluster, or with the whole grid
    // (cooperative).  Large clusters do not reach every SM (16 CTAs: 7 clusters, where 9 groups fit), but a cluster launch may
    // overlap the end of the kernel in front: taken where it needs no more rounds of row blocks.  us per call, cooperative ->
    // clusters: 1 x 512 10.3 -> 7.6, 7 x 752 10.3 -> 8.1, 24 x 1000 20.5 -> 18.5, 7 x 1536 16.4 -> 14.8; with one round more (1 x 2048)
    // 10.2 -> 10.5.
    out->clusters = false;
    if (C > 1 && C <= 16) {
        const int clusters = gridrow_max_clusters<D, OutT>(dev, C);
        if (clusters > 0 && rounds(clusters < out->n_groups ? clusters : out->n_groups) <= rounds(out->n_groups)) {
            out->clusters = true;
            if (clusters < out->n_groups) out->n_groups = clusters;
        }
    }
    if (out->n_groups > total) out->n_groups = out->total_items;
    out->longest = static_cast<uint32_t>(rounds(out->n_groups));
    return ATTNW_OK;
}
// 16-byte entries of an exchange area that serves every grid of up to `max_ctas` CTAs: the pairs of each CTA and, where the
// rows have owners (groups of more than kMaxDirectCtas), the results of each group.
constexpr size_t gridrow_entries(int max_ctas) {
    return static_cast<size_t>(max_ctas + max_ctas / (gr::kMaxDirectCtas + 1)) * gr::kXchgDepth * kTile;
}

// Returns ATTNW_ERR_UNSUPPORTED when the grid does not fit at once after all (SMs taken away from this context).
template <int D, typename OutT>
int enqueue_gridrow(const GridrowShape& g, const void* Q, const void* K, void* P, int BH, int N, float scale, uint4* xchg,
                    uint32_t tag_base, cudaStream_t stream) {
    using L = gr::Smem<D>;
    auto kernel = gr::attnw_gridrow_kernel<D, OutT>;
    CUtensorMap tm_q, tm_k, tm_p;
    int rc = encode_3d(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Q, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK)
        rc = encode_3d(&tm_p, sizeof(OutT) == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, sizeof(OutT), P,
                       N, N, BH, 128 / sizeof(OutT), 32);
    if (rc != ATTNW_OK) return rc;
    const float scale_log2e = static_cast<float>(static_cast<double>(scale) * 1.4426950408889634074);
    cudaError_t launched;
    if (g.group_ctas == 1 || g.clusters) {
        launched = launch_overlapped(kernel, static_cast<unsigned>(g.n_groups * g.group_ctas), gr::kThreads, L::kDynamicBytes, stream,
                                     g.group_ctas, tm_q, tm_k, tm_p, N, g.total_items, g.group_ctas, g.n_groups, scale_log2e, xchg,
                                     tag_base);
    } else {
        // Not overlapped: CTAs that wait for the kernel in front while another stream's cooperative grid holds the other SMs
        // could leave both grids incomplete.
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;  // every CTA of the grid is resident at once, or the launch fails
        attr[0].val.cooperative = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(gr::kThreads, 1, 1);
        cfg.gridDim = dim3(static_cast<unsigned>(g.n_groups * g.group_ctas), 1, 1);
        cfg.dynamicSmemBytes = L::kDynamicBytes;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        launched = cudaLaunchKernelEx(&cfg, kernel, tm_q, tm_k, tm_p, N, g.total_items, g.group_ctas, g.n_groups, scale_log2e, xchg, tag_base);
    }
    if (launched != cudaSuccess) {
        (void)cudaGetLastError();
        return launched == cudaErrorCooperativeLaunchTooLarge ? ATTNW_ERR_UNSUPPORTED : ATTNW_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ATTNW_OK;
}

// The exchange area that a launch on `stream` uses; called with the areas' mutex held.
int gridrow_area(GridrowAreas* areas, int sm_count, cudaStream_t stream, GridrowArea** out) {
    unsigned long long id = 0;
    if (cudaStreamGetId(stream, &id) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    for (int a = 0; a < areas->count; ++a)
        if (areas->area[a].stream_id == id) {
            *out = &areas->area[a];
            return ATTNW_OK;
        }
    // The calls below are allowed while another thread captures a stream.
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    areas->several_streams = areas->count > 0;
    int rc = ATTNW_OK;
    GridrowArea* area = nullptr;
    for (int a = 0; a < areas->count && !area; ++a)
        if (areas->area[a].recorded && cudaEventQuery(areas->area[a].last) == cudaSuccess) area = &areas->area[a];
    if (!area && areas->count < kMaxGridrowAreas) {
        GridrowArea fresh;
        const size_t bytes = gridrow_entries(sm_count) * sizeof(uint4);
        void* p = nullptr;
        // Zero, so that no entry carries a valid tag: by the stream itself, which runs the area's first launch (the legacy stream may
        // not be used while another thread captures a stream that synchronises with it, and doing so spoils that capture).
        if (cudaMalloc(&p, bytes) != cudaSuccess || cudaEventCreateWithFlags(&fresh.last, cudaEventDisableTiming) != cudaSuccess ||
            cudaMemsetAsync(p, 0, bytes, stream) != cudaSuccess) {
            if (fresh.last) cudaEventDestroy(fresh.last);
            if (p) cudaFree(p);
            rc = ATTNW_ERR_UNSUPPORTED;  // no memory for it: the caller takes a kernel that needs none
        } else {
            fresh.xchg = static_cast<uint4*>(p);
            area = &areas->area[areas->count++];
            *area = fresh;
        }
    } else if (!area) {
        for (int tries = 0; tries < kMaxGridrowAreas && !area; ++tries) {
            GridrowArea* victim = &areas->area[areas->next_victim++ % kMaxGridrowAreas];
            if (victim->recorded) area = victim;  // (all but the first stream's always are)
        }
        if (!area)
            rc = ATTNW_ERR_UNSUPPORTED;
        else if (cudaStreamWaitEvent(stream, area->last, 0) != cudaSuccess)
            rc = ATTNW_ERR_CUDA;
    }
    (void)cudaGetLastError();  // cudaErrorNotReady of the queries
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (rc != ATTNW_OK) return rc;
    area->stream_id = id;
    area->recorded = false;
    *out = area;
    return ATTNW_OK;
}

// Grid-row kernel: one CTA per SM; consecutive ceil(N / 256) CTAs, a cluster or a part of a cooperative grid, form a group that owns
// a 128-row block and walks a contiguous part of the list of row blocks.  Returns ATTNW_ERR_UNSUPPORTED when the
// device cannot hold a whole group at once, and for groups of several CTAs on a stream that is being captured.
template <int D, typename OutT>
int launch_gridrow(DeviceInfo* dev, const void* Q, const void* K, void* P, int BH, int N, float scale, cudaStream_t stream) {
    GridrowShape g;
    int rc = gridrow_shape<D, OutT>(dev, BH, N, dev->sm_count, &g);
    if (rc != ATTNW_OK) return rc;
    if (g.group_ctas == 1) return enqueue_gridrow<D, OutT>(g, Q, K, P, BH, N, scale, nullptr, 0, stream);
    // A captured launch would be replayed with the tags of its capture, at any time beside any other launch.
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    if (capture != cudaStreamCaptureStatusNone) return ATTNW_ERR_UNSUPPORTED;
    GridrowAreas& areas = g_gridrow_areas[dev - g_devices];
    std::lock_guard<std::mutex> lock(areas.mutex);
    GridrowArea* area = nullptr;
    rc = gridrow_area(&areas, dev->sm_count, stream, &area);
    if (rc != ATTNW_OK) return rc;
    uint32_t tag_base = 0;
    if (take_tags(&area->tag, g.longest, &tag_base) &&
        cudaMemsetAsync(area->xchg, 0, gridrow_entries(dev->sm_count) * sizeof(uint4), stream) != cudaSuccess) {
        (void)cudaGetLastError();
        area->tag = kLastTag;
        return ATTNW_ERR_CUDA;
    }
    rc = enqueue_gridrow<D, OutT>(g, Q, K, P, BH, N, scale, area->xchg, tag_base, stream);
    if (rc == ATTNW_OK && areas.several_streams) {
        area->recorded = cudaEventRecord(area->last, stream) == cudaSuccess;
        if (!area->recorded) rc = ATTNW_ERR_CUDA;
    }
    return rc;
}

template <int D>
int launch_attn(const void* Q, const void* K, const void* V, void* O, int BH, int N, float scale, cudaStream_t stream) {
    using L = FusedSmem<D>;
    auto kernel = av::attn_fused_kernel<D>;
    CUtensorMap tm_q, tm_k, tm_v, tm_o;
    int rc = encode_3d(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Q, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_v, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, V, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_o, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, O, D, N, BH, 64, kTile);
    if (rc != ATTNW_OK) return rc;
    if (allow_smem<av::attn_fused_kernel<D>>(L::kDynamicBytes) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    const int row_blocks = (N + kRowsPerCta - 1) / kRowsPerCta;
    const float scale_log2e = static_cast<float>(static_cast<double>(scale) * 1.4426950408889634074);
    kernel<<<static_cast<unsigned>(BH * row_blocks), kFusedThreads, L::kDynamicBytes, stream>>>(tm_q, tm_k, tm_v, tm_o, N,
                                                                                                 row_blocks, scale_log2e);
    if (cudaGetLastError() != cudaSuccess) return ATTNW_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ATTNW_OK;
}

// How many clusters of `ctas` CTAs of the one-pass attention kernel the device holds at once; -1 = none.
template <int D>
int attn_max_clusters(DeviceInfo* dev, int ctas) {
    std::atomic<int>& memo = dev->attn_clusters[D == 128][ctas];
    int n = memo.load(std::memory_order_relaxed);
    if (n != 0) return n;
    auto kernel = av1::attn_onepass_kernel<D, av1::kCluster>;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(ctas);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(av1::Smem<D>::threads(av1::kCluster), 1, 1);
    cfg.gridDim = dim3(static_cast<unsigned>(ctas * dev->sm_count), 1, 1);
    cfg.dynamicSmemBytes = av1::Smem<D>::kDynamicBytes;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (allow_smem<av1::attn_onepass_kernel<D, av1::kCluster>>(av1::Smem<D>::kDynamicBytes) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 1) {
        (void)cudaGetLastError();
        n = -1;
    }
    memo.store(n, std::memory_order_relaxed);
    return n;
}

template <int D>
int launch_attn_onepass(DeviceInfo* dev, const void* Q, const void* K, const void* V, void* O, int BH, int N, float scale, cudaStream_t stream) {
    using L = av1::Smem<D>;
    CUtensorMap tm_q, tm_k, tm_v, tm_o;
    int rc = encode_3d(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Q, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_v, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, V, D, N, BH, 64, kTile);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_o, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, O, D, N, BH, 64, kTile);
    if (rc != ATTNW_OK) return rc;
    // Two query tiles per CTA; or one whose even and odd key tiles are worked on side by side; or one for a cluster of 2 or 4 CTAs.  Chosen by
    // the rounds of key tiles on the device (about 1.6 us each at d = 64, 1.9 at d = 128, and there a tenth more where the units have key tiles
    // of their own) plus what a round of CTAs costs besides: 2.5 of them for its begin, set-up and epilogue, 2 more for a cluster's merge.  us
    // per call, one CTA -> cluster: 1 x 4744 (d = 64) 43.5 -> 28.5, 1 x 9260 (d = 128) 85.6 -> 53.6, 4 x 2155 24.2 -> 19.8, 3 x 824 11.9 ->
    // 10.8, 1 x 1000 13.3 -> 13.2.
    // Or full rounds of CTAs first, and the query tiles that are left spread over the device by a second launch.
    // One launch -> two: 2 x 10215 (d = 64, 160 query tiles) 129 -> 104, 3 x 13719 (d = 128) 312 -> 258, 22 x 1940 (d = 64) 51 -> 45, 5 x 4607
    // (d = 64) 65 -> 56, 19 x 10023 (d = 128) 1058 -> 954, 114 x 692 (d = 128) 48.7 -> 46.5; 9 x 2487 (d = 128) 37.9 -> 39.1, not taken.  The
    // second launch counts as 0.75 key tiles, and has to give 4 percent, or 8 where the number of query tiles is odd: a head's last CTA has one
    // query tile then, and the rounds of one launch overlap better than they are counted (not taken: 150 x 384, d = 64 22.2 / 23.8, 150 x 640
    // 40.1 / 43.4, 9 x 3000 45.9 / 49.9, 300 x 500, d = 128 63.1 / 65.3).  Of 836 sizes near full rounds, each measured both ways, none is more
    // than 0.5 percent behind the better one launch; with 0.5 and 3 percent for all 29 were by more than 1.5, up to 8.
    const long long tiles = (N + kTile - 1) / kTile, pairs = (tiles + 1) / 2, all = BH * tiles;
    const int sms = dev->sm_count;
    struct Part {
        av1::Mode mode;
        int ctas;         // per query tile (kWhole: per pair of query tiles)
        long long first;  // query tile (pair of them) of all heads that the part begins with, and how many it has
        long long count;
        double cost;
    };
    auto waves = [](long long work, long long at_once) { return static_cast<double>((work + at_once - 1) / at_once); };
    const double whole_round = static_cast<double>(tiles) + 2.5, own = D == 128 ? 1.1 : 1.0, split_round = (static_cast<double>(pairs) + 2.5) * own;
    auto best_part = [&](long long first_tile) {  // for the query tiles from there on, each by a CTA or a cluster
        const long long n = all - first_tile;
        Part p{av1::kSplit, 1, first_tile, n, waves(n, sms) * split_round};
        for (int g = 2; g <= av1::kMaxCluster && 2 * g <= tiles && all * g <= INT_MAX; g *= 2) {
            const int clusters = attn_max_clusters<D>(dev, g);
            if (clusters < 1) break;
            const double c = waves(n, clusters) * (static_cast<double>((tiles + 2 * g - 1) / (2 * g)) + 4.5) * own;
            if (c * 1.05 < p.cost) p = {av1::kCluster, g, first_tile, n, c};
        }
        return p;
    };
    Part parts[2] = {{av1::kWhole, 1, 0, BH * pairs, waves(BH * pairs, sms) * whole_round}, {}};
    int n_parts = 1;
    double best = parts[0].cost;
    if (tiles > 1 && all <= INT_MAX) {
        const Part one = best_part(0);
        if (one.cost * 1.05 < best) {
            parts[0] = one;
            best = one.cost;
        }
        for (const av1::Mode mode : {av1::kWhole, av1::kSplit}) {
            const long long units = mode == av1::kWhole ? BH * pairs : all, full = units / sms * sms;
            if (full == 0 || full == units) continue;
            const double front = static_cast<double>(full / sms) * (mode == av1::kWhole ? whole_round : split_round);
            const Part rest = best_part(mode == av1::kWhole ? full / pairs * tiles + 2 * (full % pairs) : full);
            const double cost = front + rest.cost + 0.75;
            if (cost * (tiles % 2 == 0 ? 1.04 : 1.08) < best) {
                parts[0] = {mode, 1, 0, full, front};
                parts[1] = rest;
                n_parts = 2;
                best = cost;
            }
        }
    }
    const float scale_log2e = static_cast<float>(static_cast<double>(scale) * 1.4426950408889634074);
    for (int i = 0; i < n_parts; ++i) {
        const Part& p = parts[i];
        const cudaError_t allowed = p.mode == av1::kWhole   ? allow_smem<av1::attn_onepass_kernel<D, av1::kWhole>>(L::kDynamicBytes)
                                    : p.mode == av1::kSplit ? allow_smem<av1::attn_onepass_kernel<D, av1::kSplit>>(L::kDynamicBytes)
                                                            : allow_smem<av1::attn_onepass_kernel<D, av1::kCluster>>(L::kDynamicBytes);
        auto kernel = p.mode == av1::kWhole   ? av1::attn_onepass_kernel<D, av1::kWhole>
                      : p.mode == av1::kSplit ? av1::attn_onepass_kernel<D, av1::kSplit>
                                              : av1::attn_onepass_kernel<D, av1::kCluster>;
        if (allowed != cudaSuccess ||
            launch_overlapped(kernel, static_cast<unsigned>(p.count * p.ctas), L::threads(p.mode), L::kDynamicBytes, stream, p.ctas, tm_q, tm_k,
                              tm_v, tm_o, N, static_cast<int>(p.mode == av1::kWhole ? pairs : tiles), scale_log2e, static_cast<__nv_bfloat16*>(O),
                              p.ctas, static_cast<int>(p.first)) != cudaSuccess) {
            (void)cudaGetLastError();
            return ATTNW_ERR_CUDA;
        }
        g_launches.fetch_add(1, std::memory_order_relaxed);
    }
    return ATTNW_OK;
}

// Host-only checks of the attention call; no CUDA call is made here.
int validate_attn(const void* Q, const void* K, const void* V, const void* O, int B, int H, int N, int d, float scale) {
    if (!Q || !K || !V || !O) return ATTNW_ERR_NULL_POINTER;
    if (B < 1 || H < 1 || N < 1 || d < 1) return ATTNW_ERR_BAD_SHAPE;
    if (!(scale >= 0.0f) || !std::isfinite(scale)) return ATTNW_ERR_BAD_SHAPE;
    const long long bh = static_cast<long long>(B) * H;
    if (bh > INT_MAX) return ATTNW_ERR_BAD_SHAPE;
    if (bh * ((static_cast<long long>(N) + kRowsPerCta - 1) / kRowsPerCta) > INT_MAX) return ATTNW_ERR_BAD_SHAPE;
    if (N > (1 << 24)) return ATTNW_ERR_BAD_SHAPE;
    if (d != 64 && d != 128) return ATTNW_ERR_UNSUPPORTED;
    if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(O)) return ATTNW_ERR_MISALIGNED;
    const unsigned long long bytes = static_cast<unsigned long long>(bh) * N * d * 2ull;
    if (overlaps(O, bytes, Q, bytes) || overlaps(O, bytes, K, bytes) || overlaps(O, bytes, V, bytes)) return ATTNW_ERR_ALIASING;
    return ATTNW_OK;
}

// Host-only checks of the projection call; no CUDA call is made here.
int validate_project(const void* X, const void* Wq, const void* Wk, const void* Q, const void* K, int B, int N, int d_model,
                     int H, int d) {
    if (!X || !Wq || !Wk || !Q || !K) return ATTNW_ERR_NULL_POINTER;
    if (B < 1 || N < 1 || d_model < 1 || H < 1 || d < 1) return ATTNW_ERR_BAD_SHAPE;
    if (N > (1 << 24) || d_model > (1 << 20)) return ATTNW_ERR_BAD_SHAPE;  // keeps every tensor-map stride below 2^40 bytes
    const long long bh = static_cast<long long>(B) * H;
    if (bh > INT_MAX || static_cast<long long>(H) * d > INT_MAX) return ATTNW_ERR_BAD_SHAPE;
    const long long col_tiles = (static_cast<long long>(H) * d + 127) / 128;  // the smallest tiles the call may be cut into
    const long long row_tiles = (static_cast<long long>(N) + 127) / 128;
    if (2 * col_tiles * row_tiles > INT_MAX / B) return ATTNW_ERR_BAD_SHAPE;
    if (d != 64 && d != 128) return ATTNW_ERR_UNSUPPORTED;
    if (d_model % 8 != 0) return ATTNW_ERR_MISALIGNED;  // rows of X and of the weights must start on 16-byte boundaries
    if (!aligned16(X) || !aligned16(Wq) || !aligned16(Wk) || !aligned16(Q) || !aligned16(K)) return ATTNW_ERR_MISALIGNED;
    const unsigned long long x_bytes = static_cast<unsigned long long>(B) * N * d_model * 2ull;
    const unsigned long long w_bytes = static_cast<unsigned long long>(H) * d * d_model * 2ull;
    const unsigned long long o_bytes = static_cast<unsigned long long>(bh) * N * d * 2ull;
    if (overlaps(Q, o_bytes, K, o_bytes)) return ATTNW_ERR_ALIASING;
    for (const void* out : {Q, K})
        if (overlaps(out, o_bytes, X, x_bytes) || overlaps(out, o_bytes, Wq, w_bytes) || overlaps(out, o_bytes, Wk, w_bytes))
            return ATTNW_ERR_ALIASING;
    return ATTNW_OK;
}

int launch_project(const DeviceInfo* dev, const void* X, const void* Wq, const void* Wk, void* Q, void* K, int B, int N, int d_model,
                   int H, int d, cudaStream_t stream) {
    CUtensorMap tm_x, tm_wq, tm_wk, tm_q, tm_k;
    const uint64_t hd = static_cast<uint64_t>(H) * d, bh = static_cast<uint64_t>(B) * H;
    int rc = encode_3d(&tm_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, X, d_model, N, B, proj::kKSlice, proj::kRows);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_wq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Wq, d_model, hd, 1, proj::kKSlice, proj::kFeatures / 2);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_wk, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Wk, d_model, hd, 1, proj::kKSlice, proj::kFeatures / 2);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Q, d, N, bh, 64, 32);
    if (rc == ATTNW_OK) rc = encode_3d(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, K, d, N, bh, 64, 32);
    if (rc != ATTNW_OK) return rc;
    auto launch = [&](auto pair, int workers, int block, int whole) -> int {
        constexpr bool kPair = decltype(pair)::value;
        constexpr int kCtas = kPair ? 2 : 1;
        if (allow_smem<proj::project_qk_kernel<kPair>>(proj::kDynamicBytes) != cudaSuccess ||
            launch_overlapped(proj::project_qk_kernel<kPair>, kCtas * static_cast<unsigned>(workers), proj::kThreads, proj::kDynamicBytes, stream, kCtas,
                              tm_x, tm_wq, tm_wk, tm_q, tm_k, B, N, d_model, H, d, block, whole) != cudaSuccess) {
            (void)cudaGetLastError();
            return ATTNW_ERR_CUDA;
        }
        g_launches.fetch_add(1, std::memory_order_relaxed);
        return ATTNW_OK;
    };
    // One CTA a tile of 128 x 128, without a partner, where one round of them holds the call and either a few slices are all there is - a pair's
    // set-up and end cost it 0.2 to 0.4 us - or narrow tiles by pairs would not be one round (an odd number of row blocks, most often one or three:
    // whole tiles leave half of the SMs idle then).  us per call, pairs -> single CTAs: 2 x 64 x 256 to 4 x 64 4.70 -> 4.52, 1 x 128 x 64 to 8 x 64
    // 4.27 -> 3.96, 1 x 384 x 64 to 40 x 64 5.03 -> 4.02, 1 x 300 x 1024 to 40 x 64 9.68 -> 7.39, 1 x 128 x 2048 to 96 x 64 15.2 -> 12.2, 1 x 600 x
    // 4096 to 28 x 64 23.4 -> 18.3; but 1 x 1000 x 512 to 16 x 64 5.53 -> 5.61, 1 x 1000 x 4096 to 16 x 64 14.8 -> 17.3 (a pair fetches 24 KB a
    // slice, not 32), and a few rows of X, which all CTAs read from the same places of L2, want fewer readers: 1 x 8 x 4096 to 80 x 64 24.1 -> 32.4,
    // 1 x 16 x 4096 23.5 -> 20.7.
    // The same with tiles of 128 x 256, where pairs need a second round for what single CTAs do in one: 1 x 300 x 768 to 40 x 128 10.4 -> 8.4, 1 x
    // 1400 x 2048 to 13 x 128 22.6 -> 15.7, 1 x 128 x 768 to 80 x 128 12.3 -> 8.4, 1 x 64 x 4096 to 148 x 128 58.2 -> 53.4.
    constexpr int kNarrow = proj::kFeatures / 2, kWide = proj::kFeatures;
    auto tiles_of = [&](int block, int ctas) { return proj::Grid(B, N, static_cast<int>(hd), block, ctas).tiles(); };
    const int sms = dev->sm_count, pairs = sms / 2;
    const bool narrow = tiles_of(kNarrow, 2) <= pairs, shared_x = d_model > 512 && static_cast<long long>(B) * N < 64 && static_cast<long long>(B) * N * d_model < 65536;
    if (tiles_of(kNarrow, 1) <= sms && (d_model <= 256 || (!narrow && !shared_x)))
        return launch(std::false_type{}, tiles_of(kNarrow, 1), kNarrow, tiles_of(kNarrow, 1));
    if (tiles_of(kWide, 1) <= sms && tiles_of(kWide, 2) > pairs && !shared_x) return launch(std::false_type{}, tiles_of(kWide, 1), kWide, tiles_of(kWide, 1));
    // Tiles of 256 x 256 per pair of CTAs; narrow ones of 256 x 128 where a single round of them holds the call, since a narrow slice still takes
    // 0.6 to 0.75 of the time of a whole one (X's rows are fetched for half of the MMAs).  A last round whose tiles would occupy at most
    // half of the pairs takes them cut in two.  us per call, whole tiles only -> as chosen: narrow 4 x 100 x 1536 to 12 x 128 11.3 -> 7.7,
    // 1 x 1000 x 1024 to 16 x 64 9.3 -> 6.7, 2 x 949 x 576 to 9 x 64 7.2 -> 5.7, 1 x 256 x 4096 to 64 x 64 24.9 -> 21.2; tiles cut in two 1 x 2048 x
    // 4096 to 32 x 128 (256 tiles for 74 pairs) 111.8 -> 107.6, 2 x 444 x 3200 to 25 x 128 (100) 40.7 -> 37.4, 4 x 3749 x 4080 to 10 x 64 (300) 142.5 -> 140.8.
    const int block = narrow ? kNarrow : kWide;
    const int tiles = tiles_of(block, 2), last = tiles % pairs;
    const int whole = block == kWide && 2 * last <= pairs ? tiles - last : tiles;
    const int items = 2 * tiles - whole;
    return launch(std::true_type{}, items < pairs ? items : pairs, block, whole);
}

// Whether the choice by shape takes the grid-row kernel for rows of N keys: it computes every score and exponential once, the
// two-pass kernel twice, but groups of ceil(N / 256) CTAs leave SMs idle, and the exchange grows with the group.
// A 128 x 256 block costs it some 4450 cycles of an SM against 6000: it pays while two thirds of the SMs have work.
// Measured on B200, us per call, two-pass -> grid-row, B*H x N (CTAs a group, SMs in use): bfloat16 2 x 6000 (24, 144)
// 132 -> 39, 8 x 8192 (32, 128) 428 -> 319, 2 x 13000 (51, 102) 319 -> 233, 8 x 16384 (64, 128) 1551 -> 1212, 1 x 25600
// (100, 100) 601 -> 425, 1 x 32768 (128, 128) 780 -> 803; float32 2 x 512 16.4 -> 10.2, 16 x 2052 112 -> 80, 32 x 4096
// 613 -> 492, 2 x 13000 399 -> 355, 1 x 25600 776 -> 726, 1 x 32768 1193 -> 1254.
bool gridrow_pays(const DeviceInfo* dev, int N) {
    const int group_ctas = (N + gr::kSlabCols - 1) / gr::kSlabCols;
    return group_ctas <= 112 && dev->sm_count / group_ctas * group_ctas * 3 >= dev->sm_count * 2;
}

// Enqueues `first` and `second` on a stream that is being captured as two branches of its graph, which may run side by side.  By
// the capture's own dependencies and not by a second stream: a stream belongs to one capture until that ends, so two captures
// open at once could not share it.
template <typename First, typename Second>
int capture_side_by_side(cudaStream_t s, First first, Second second) {
    constexpr size_t kMost = 16;
    cudaGraphNode_t before[kMost], behind_first[kMost];
    auto dependencies = [s](cudaGraphNode_t* out, size_t* n) {
        cudaStreamCaptureStatus status;
        const cudaGraphNode_t* nodes = nullptr;
        if (cudaStreamGetCaptureInfo(s, &status, nullptr, nullptr, &nodes, n) != cudaSuccess || *n > kMost) {
            (void)cudaGetLastError();
            return false;
        }
        for (size_t i = 0; i < *n; ++i) out[i] = nodes[i];
        return true;
    };
    size_t n_before = 0, n_first = 0;
    const bool known = dependencies(before, &n_before);
    int rc = first(s);
    if (rc != ATTNW_OK) return rc;
    if (!known || !dependencies(behind_first, &n_first)) return second(s);  // one behind the other
    if (cudaStreamUpdateCaptureDependencies(s, before, n_before, cudaStreamSetCaptureDependencies) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    rc = second(s);
    if (cudaStreamUpdateCaptureDependencies(s, behind_first, n_first, cudaStreamAddCaptureDependencies) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    return rc;
}

template <typename OutT>
int fused_entry(const void* Q, const void* K, void* P, int B, int H, int N, int d, float scale, void* stream) {
    int rc = validate_fused(Q, K, P, B, H, N, d, scale, sizeof(OutT));
    if (rc != ATTNW_OK) return rc;
    DeviceInfo* dev = nullptr;
    rc = current_device(&dev);
    if (rc != ATTNW_OK) return rc;
    rc = load_encoder();
    if (rc != ATTNW_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int variant = g_fused_variant.load(std::memory_order_relaxed);
    const bool resident_fits = sizeof(OutT) == 2 && N <= kResidentMaxN;
    if ((variant == 2 || variant == 3) && !resident_fits) return ATTNW_ERR_UNSUPPORTED;
    if (variant == 4) {
        if constexpr (sizeof(OutT) == 2) {
            if (N > gr::kMaxN) return ATTNW_ERR_UNSUPPORTED;
            return (d == 64) ? launch_gridrow<64, OutT>(dev, Q, K, P, B * H, N, scale, s)
                             : launch_gridrow<128, OutT>(dev, Q, K, P, B * H, N, scale, s);
        }
        return ATTNW_ERR_UNSUPPORTED;
    }
    if (variant == 3) {
        if constexpr (sizeof(OutT) == 2)
            return (d == 64) ? launch_resident<64>(dev, Q, K, P, B * H, N, scale, s, true)
                             : launch_resident<128>(dev, Q, K, P, B * H, N, scale, s, true);
        return ATTNW_ERR_UNSUPPORTED;
    }
    // Choice by shape, first candidate: the grid-row kernel, where its groups fit the device well (see gridrow_pays).
    // A device that cannot hold a whole group at once falls through to the older choice.
    if (variant == 0 && gridrow_pays(dev, N)) {
        rc = (d == 64) ? launch_gridrow<64, OutT>(dev, Q, K, P, B * H, N, scale, s)
                       : launch_gridrow<128, OutT>(dev, Q, K, P, B * H, N, scale, s);
        if (rc != ATTNW_ERR_UNSUPPORTED) return rc;
    }
    // Older choice by shape: the resident kernel whenever it can serve the call.  It spreads one 128-row block over the
    // C SMs of a cluster, so it also fills the device when B*H is small (B*H = 1, N = 4096, d = 128: 25 us
    // against 96 us; B*H = 12, N = 2048, d = 64: 37 against 51 us); between B*H = 8 and 16 at N = 4096 the
    // two kernels are within 2 % of each other, above that the resident kernel leads again.
    // Clusters of more than 8 CTAs (N > 4096) fit only 7 times (112 SMs): there the two-pass kernel with two CTAs per
    // row block is ahead except for a single head (B*H = 4, N = 8192: 188 against 221 us), so the choice by shape
    // stops at N = 4096; variant 2 serves N <= 8192 on request.
    const bool resident_pays = N <= 8 * kSlab;
    if (resident_fits && (variant == 2 || (variant == 0 && resident_pays))) {
        if constexpr (sizeof(OutT) == 2) {
            // Clusters of 8 cannot occupy every SM (15 x 8 = 120 of 148 on B200).  When the call is chosen by
            // shape, the heads are split: the resident kernel takes most of them on the caller's stream, and
            // the two-pass kernel, forked onto a side stream, works through the rest on the SMs the clusters
            // leave idle; the caller's stream joins before the call's work counts as done.
            const int cluster_ctas = (N + kSlab - 1) / kSlab;
            const int clusters = (d == 64) ? resident_max_clusters<64>(dev, cluster_ctas)
                                           : resident_max_clusters<128>(dev, cluster_ctas);
            const int bh = B * H;
            const int idle_sms = clusters > 0 ? dev->sm_count - clusters * cluster_ctas : 0;
            int bh_two_pass = 0;
            if (variant == 0 && idle_sms >= 8 && bh >= 8) {
                // Cost model in units of one resident row block: a cluster finishes one row block per unit, a
                // two-pass CTA (256 rows on one SM) takes 2 * C / kTwoPassPerSm units, both in whole waves.
                const long long blocks_per_head = (N + kTile - 1) / kTile;
                const long long ctas_per_head = (N + kRowsPerCta - 1) / kRowsPerCta;
                const double cta_units = 2.0 * cluster_ctas / kTwoPassPerSm;
                double best = static_cast<double>((bh * blocks_per_head + clusters - 1) / clusters);
                for (int cand = 1; cand <= bh / 2; ++cand) {
                    const double t_res = static_cast<double>(((bh - cand) * blocks_per_head + clusters - 1) / clusters);
                    const double t_two = static_cast<double>((cand * ctas_per_head + idle_sms - 1) / idle_sms) * cta_units;
                    const double t = t_res > t_two ? t_res : t_two;
                    if (t < best) {
                        best = t;
                        bh_two_pass = cand;
                    }
                }
            }
            if (bh_two_pass > 0) {
                const int bh_res = bh - bh_two_pass;
                const size_t qk_off = static_cast<size_t>(bh_res) * N * d * 2;
                const size_t p_off = static_cast<size_t>(bh_res) * N * N * 2;
                const char* q2 = static_cast<const char*>(Q) + qk_off;
                const char* k2 = static_cast<const char*>(K) + qk_off;
                char* p2 = static_cast<char*>(P) + p_off;
                auto resident = [&](cudaStream_t on) {
                    return (d == 64) ? launch_resident<64>(dev, Q, K, P, bh_res, N, scale, on)
                                     : launch_resident<128>(dev, Q, K, P, bh_res, N, scale, on);
                };
                auto two_pass = [&](cudaStream_t on) {
                    return (d == 64) ? launch_fused<64, OutT>(dev, q2, k2, p2, bh_two_pass, N, scale, on, false)
                                     : launch_fused<128, OutT>(dev, q2, k2, p2, bh_two_pass, N, scale, on, false);
                };
                cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
                if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
                    (void)cudaGetLastError();
                    return ATTNW_ERR_CUDA;
                }
                if (capture != cudaStreamCaptureStatusNone) return capture_side_by_side(s, resident, two_pass);
                std::lock_guard<std::mutex> lock(g_split_mutex);
                if (!dev->side_stream) {
                    if (cudaStreamCreateWithFlags(&dev->side_stream, cudaStreamNonBlocking) != cudaSuccess ||
                        cudaEventCreateWithFlags(&dev->fork_event, cudaEventDisableTiming) != cudaSuccess ||
                        cudaEventCreateWithFlags(&dev->join_event, cudaEventDisableTiming) != cudaSuccess) {
                        (void)cudaGetLastError();
                        return ATTNW_ERR_CUDA;
                    }
                }
                if (cudaEventRecord(dev->fork_event, s) != cudaSuccess) return ATTNW_ERR_CUDA;
                rc = resident(s);
                if (rc != ATTNW_OK) return rc;
                if (cudaStreamWaitEvent(dev->side_stream, dev->fork_event, 0) != cudaSuccess) return ATTNW_ERR_CUDA;
                rc = two_pass(dev->side_stream);
                if (cudaEventRecord(dev->join_event, dev->side_stream) != cudaSuccess ||
                    cudaStreamWaitEvent(s, dev->join_event, 0) != cudaSuccess)
                    return ATTNW_ERR_CUDA;
                return rc;
            }
        }
        rc = (d == 64) ? launch_resident<64>(dev, Q, K, P, B * H, N, scale, s)
                       : launch_resident<128>(dev, Q, K, P, B * H, N, scale, s);
        if (rc != ATTNW_ERR_UNSUPPORTED || variant == 2) return rc;  // no cluster of that size here: two-pass
    }
    if (d == 64) return launch_fused<64, OutT>(dev, Q, K, P, B * H, N, scale, s);
    return launch_fused<128, OutT>(dev, Q, K, P, B * H, N, scale, s);
}

int validate_rows(const void* S, const void* P, long long rows, long long cols, size_t p_esize, bool allow_inplace) {
    if (!S || !P) return ATTNW_ERR_NULL_POINTER;
    if (rows < 1 || cols < 1) return ATTNW_ERR_BAD_SHAPE;
    if (cols > (1ll << 40) || rows > (1ll << 40) || rows > (1ll << 62) / cols) return ATTNW_ERR_BAD_SHAPE;
    if (cols % 4 != 0) return ATTNW_ERR_MISALIGNED;
    if (!aligned16(S) || !aligned16(P)) return ATTNW_ERR_MISALIGNED;
    const unsigned long long n = static_cast<unsigned long long>(rows) * static_cast<unsigned long long>(cols);
    if (overlaps(S, n * 4ull, P, n * p_esize) && !(allow_inplace && S == P)) return ATTNW_ERR_ALIASING;
    return ATTNW_OK;
}

template <typename OutT>
int rows_entry(const void* S, void* P, long long rows, long long cols, void* stream) {
    int rc = validate_rows(S, P, rows, cols, sizeof(OutT), sizeof(OutT) == 4);
    if (rc != ATTNW_OK) return rc;
    DeviceInfo* dev = nullptr;
    rc = current_device(&dev);
    if (rc != ATTNW_OK) return rc;
    const int variant = g_rows_variant.load(std::memory_order_relaxed);
    if (variant == 3 && cols > kSoftmaxRowsRegTierMaxCols) return ATTNW_ERR_UNSUPPORTED;
    if (variant == 1 && cols > srs::kMaxCols) return ATTNW_ERR_UNSUPPORTED;
    // Longer rows can be kept in the shared memory of a CTA or of a cluster (caching form).  By default that is done
    // where it is the faster way (measured): from 8192 columns on - there the register tier needs a whole CTA of 1024
    // threads per row and stops overlapping rows - with one CTA, or a cluster of two up to 32768 columns; beyond, the two-read kernel and
    // the registers of a cluster are ahead (us, default / a cluster of two, bfloat16 6000 x 36864 241 / 252, 5000 x 45000 229 / 248; float32 308 / 298,
    // 291 / 293, 100 x 36864 6.9 / 8.9; larger clusters 1.3 to 1.9 times the default).
    const int smem_ctas = cols > kSoftmaxRowsSmemTierMinCols ? srs::cluster_ctas_for(cols) : 0;
    const bool smem_default = smem_ctas == 1 || (smem_ctas == 2 && cols <= kSoftmaxRowsRegTierMaxCols);
    if ((variant == 0 && smem_default) || (variant == 1 && smem_ctas >= 1)) {
        if (srs::launch<OutT>(static_cast<const float*>(S), static_cast<OutT*>(P), rows, cols, dev->sm_count,
                              static_cast<cudaStream_t>(stream)) == cudaSuccess) {
            g_launches.fetch_add(1, std::memory_order_relaxed);
            return ATTNW_OK;
        }
        (void)cudaGetLastError();  // no cluster of that size on this device: fall through to the two-read kernel
        if (variant == 1) return ATTNW_ERR_UNSUPPORTED;
    }
    // Rows of 43009 to 262144 columns, and from 32769 where rows are few: kept in the registers of a cluster, one read and
    // one write per element.  With many rows of up to 43008 columns the slices of a cluster of three are short and the two-read
    // kernel is ahead (6000 x 36864: 256 against 269 us, x 40960: 277 against 292, x 45000: 357 against 315); with few it has one CTA a
    // row where the clusters have three SMs.  us, two-read / cluster: bfloat16 10, 37, 49, 74, 148 x 36864 6.1 / 5.0, 6.2 / 5.1, 6.3 / 6.2,
    // 6.3 / 6.5, 7.1 / 9.4, x 43008 6.9 / 5.1, 7.0 / 5.2, 7.0 / 6.4, 7.1 / 6.7, 8.3 / 9.8; float32 37, 49 x 32772 6.4 / 5.7, 6.4 / 7.3.
    const bool few_rows = cols > kSoftmaxRowsRegTierMaxCols && rows <= dev->sm_count / 4;
    if (variant == 0 && (cols > kSoftmaxRowsRegClusterMinCols || few_rows) && cols <= srs::kRcMaxCols) {
        const int C = srs::rc_cluster_ctas_for(cols);
        const cudaError_t ce = srs::launch_regcluster<OutT>(static_cast<const float*>(S), static_cast<OutT*>(P), rows, cols,
                                                            &dev->rc_clusters[sizeof(OutT) == 4][C],
                                                            static_cast<cudaStream_t>(stream));
        if (ce == cudaSuccess) {
            g_launches.fetch_add(1, std::memory_order_relaxed);
            return ATTNW_OK;
        }
        (void)cudaGetLastError();  // no cluster of that size on this device: the two-read kernel
    }
    cudaError_t e = softmax_rows_launch<OutT>(static_cast<const float*>(S), static_cast<OutT*>(P), rows, cols,
                                              dev->sm_count, static_cast<cudaStream_t>(stream), variant == 3 ? 1 : (variant == 2 ? 2 : 0));
    if (e != cudaSuccess) return ATTNW_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ATTNW_OK;
}

// ---- host-buffer entry points: staging buffers kept per device, two streams ---------------
struct HostStaging {
    void* buf[2][3] = {{nullptr, nullptr, nullptr}, {nullptr, nullptr, nullptr}};
    size_t cap[2][3] = {{0, 0, 0}, {0, 0, 0}};
    cudaStream_t stream[2] = {nullptr, nullptr};
    bool streams_ready = false;
};
HostStaging g_staging[kMaxDevices];

int staging_for_current_device(HostStaging** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ATTNW_ERR_CUDA;
    HostStaging& st = g_staging[dev];
    if (!st.streams_ready) {
        for (int i = 0; i < 2; ++i)
            if (cudaStreamCreateWithFlags(&st.stream[i], cudaStreamNonBlocking) != cudaSuccess) return ATTNW_ERR_CUDA;
        st.streams_ready = true;
    }
    *out = &st;
    return ATTNW_OK;
}

int staging_reserve(HostStaging* st, int slot, int which, size_t bytes) {
    if (st->cap[slot][which] >= bytes) return ATTNW_OK;
    if (st->buf[slot][which]) {
        // The slot's stream may still be using the old buffer.
        if (cudaStreamSynchronize(st->stream[slot]) != cudaSuccess) return ATTNW_ERR_CUDA;
        cudaFree(st->buf[slot][which]);
        st->buf[slot][which] = nullptr;
        st->cap[slot][which] = 0;
    }
    if (cudaMalloc(&st->buf[slot][which], bytes) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    st->cap[slot][which] = bytes;
    return ATTNW_OK;
}

constexpr unsigned long long kHostChunkBytes = 256ull << 20;  // target size of one staged piece of P

// ---- attnw_fused_noalloc: the grid-row kernel with its exchange area in a static device array ----------------
// Scratch of the entry point that allocates nothing: the exchange area of the grid-row kernel for a grid of up to
// kNoAllocMaxCtas CTAs (messages of 16 bytes: [CTA or group][8 row blocks][128 rows]) = 3 MiB, held by every
// GPU that loads the library until the process exits.  In host code this name is only a stand-in for the symbol:
// the device address comes from cudaGetSymbolAddress (noalloc_setup below) and is what the kernel is given.
constexpr int kNoAllocMaxCtas = 160;
static __device__ __align__(256) uint4 g_noalloc_xchg[gridrow_entries(kNoAllocMaxCtas)];

struct NoAllocState {
    bool ready = false;
    uint4* xchg = nullptr;   // device address of g_noalloc_xchg on this device
    uint32_t tag = 0;        // next unused message tag of this device's array
};
NoAllocState g_noalloc[kMaxDevices];

// Once per device, with that device current.  Returns an attnw_status.
int noalloc_setup(NoAllocState** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    std::lock_guard<std::mutex> lock(g_mutex);
    NoAllocState& st = g_noalloc[dev];
    if (!st.ready) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_xchg) != cudaSuccess || ptr == nullptr) {
            (void)cudaGetLastError();
            return ATTNW_ERR_CUDA;
        }
        st.xchg = static_cast<uint4*>(ptr);
        st.tag = 0;  // the array is zero when the module is loaded, and zero is never a tag
        st.ready = true;
    }
    *out = &st;
    return ATTNW_OK;
}

template <int D>
int launch_gridrow_noalloc(DeviceInfo* dev, NoAllocState* st, const void* Q, const void* K, void* P, int BH, int N, float scale,
                           cudaStream_t stream) {
    // one CTA per SM, whole groups only, and never more CTAs than the static array has entries for
    GridrowShape g;
    int rc = gridrow_shape<D, __nv_bfloat16>(dev, BH, N, dev->sm_count < kNoAllocMaxCtas ? dev->sm_count : kNoAllocMaxCtas, &g);
    if (rc != ATTNW_OK) return rc;
    uint32_t tag_base = 0;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess) {
            (void)cudaGetLastError();
            return ATTNW_ERR_CUDA;
        }
        // A captured launch has tags that no uncaptured one uses, and repeats them, like the graph's other launches, from an array
        // that it clears first.
        const bool captured = capture != cudaStreamCaptureStatusNone;
        const bool start_over = !captured && take_tags(&st->tag, g.longest, &tag_base);
        if (captured) tag_base = kCapturedTagBase;
        if ((captured || start_over) && cudaMemsetAsync(st->xchg, 0, sizeof(g_noalloc_xchg), stream) != cudaSuccess) {
            (void)cudaGetLastError();
            if (start_over) st->tag = kLastTag;
            return ATTNW_ERR_CUDA;
        }
    }
    const int launched = enqueue_gridrow<D, __nv_bfloat16>(g, Q, K, P, BH, N, scale, st->xchg, tag_base, stream);
    return launched == ATTNW_ERR_UNSUPPORTED ? ATTNW_ERR_CUDA : launched;
}

}  // namespace

extern "C" {

int attn_fused(const void* Q, const void* K, const void* V, void* O, int B, int H, int N, int d, float scale,
               void* stream) {
    int rc = validate_attn(Q, K, V, O, B, H, N, d, scale);
    if (rc != ATTNW_OK) return rc;
    DeviceInfo* dev = nullptr;
    rc = current_device(&dev);
    if (rc != ATTNW_OK) return rc;
    rc = load_encoder();
    if (rc != ATTNW_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (g_attn_variant.load(std::memory_order_relaxed) == 1)
        return d == 64 ? launch_attn<64>(Q, K, V, O, B * H, N, scale, s) : launch_attn<128>(Q, K, V, O, B * H, N, scale, s);
    return d == 64 ? launch_attn_onepass<64>(dev, Q, K, V, O, B * H, N, scale, s)
                   : launch_attn_onepass<128>(dev, Q, K, V, O, B * H, N, scale, s);
}

int attnw_project_qk(const void* X, const void* Wq, const void* Wk, void* Q, void* K, int B, int N, int d_model, int H, int d,
                     void* stream) {
    int rc = validate_project(X, Wq, Wk, Q, K, B, N, d_model, H, d);
    if (rc != ATTNW_OK) return rc;
    DeviceInfo* dev = nullptr;
    rc = current_device(&dev);
    if (rc != ATTNW_OK) return rc;
    rc = load_encoder();
    if (rc != ATTNW_OK) return rc;
    return launch_project(dev, X, Wq, Wk, Q, K, B, N, d_model, H, d, static_cast<cudaStream_t>(stream));
}

int attnw_set_rows_variant(int variant) {
    if (variant < 0 || variant > 3) return ATTNW_ERR_BAD_SHAPE;
    g_rows_variant.store(variant, std::memory_order_relaxed);
    return ATTNW_OK;
}

int attnw_set_attn_variant(int variant) {
    if (variant < 0 || variant > 2) return ATTNW_ERR_BAD_SHAPE;
    g_attn_variant.store(variant, std::memory_order_relaxed);
    return ATTNW_OK;
}

int attnw_fused(const void* Q, const void* K, void* P, int B, int H, int N, int d, float scale, void* stream) {
    return fused_entry<__nv_bfloat16>(Q, K, P, B, H, N, d, scale, stream);
}

int attnw_fused_noalloc(const void* Q, const void* K, void* P, int B, int H, int N, int d, float scale, void* stream) {
    int rc = validate_fused(Q, K, P, B, H, N, d, scale, 2);
    if (rc != ATTNW_OK) return rc;
    if (N > gr::kMaxN) return ATTNW_ERR_UNSUPPORTED;  // beyond what the static exchange area and one group can serve
    NoAllocState* st = nullptr;
    rc = noalloc_setup(&st);
    if (rc != ATTNW_OK) return rc;
    DeviceInfo* dev = nullptr;
    rc = current_device(&dev);
    if (rc != ATTNW_OK) return rc;
    rc = load_encoder();
    if (rc != ATTNW_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return d == 64 ? launch_gridrow_noalloc<64>(dev, st, Q, K, P, B * H, N, scale, s)
                   : launch_gridrow_noalloc<128>(dev, st, Q, K, P, B * H, N, scale, s);
}

int attnw_fused_f32(const void* Q, const void* K, void* P, int B, int H, int N, int d, float scale, void* stream) {
    return fused_entry<float>(Q, K, P, B, H, N, d, scale, stream);
}

int softmax_rows(const void* S, void* P, long long rows, long long cols, void* stream) {
    return rows_entry<__nv_bfloat16>(S, P, rows, cols, stream);
}

int softmax_rows_f32(const void* S, void* P, long long rows, long long cols, void* stream) {
    return rows_entry<float>(S, P, rows, cols, stream);
}

int attnw_fused_host(const void* Q, const void* K, void* P, int B, int H, int N, int d, float scale, int p_is_f32) {
    const size_t esize = p_is_f32 ? 4 : 2;
    if (!Q || !K || !P) return ATTNW_ERR_NULL_POINTER;
    if (B < 1 || H < 1 || N < 1 || d < 1) return ATTNW_ERR_BAD_SHAPE;
    if (d != 64 && d != 128) return ATTNW_ERR_UNSUPPORTED;
    const long long bh = static_cast<long long>(B) * H;
    if (bh > INT_MAX || N > (1 << 24)) return ATTNW_ERR_BAD_SHAPE;
    if (!(scale >= 0.0f) || !std::isfinite(scale)) return ATTNW_ERR_BAD_SHAPE;
    if ((static_cast<unsigned long long>(N) * esize) % 16 != 0) return ATTNW_ERR_MISALIGNED;  // before anything is queued
    HostStaging* st = nullptr;
    int rc = staging_for_current_device(&st);
    if (rc != ATTNW_OK) return rc;
    const unsigned long long p_head = static_cast<unsigned long long>(N) * N * esize;
    const unsigned long long qk_head = static_cast<unsigned long long>(N) * d * 2ull;
    long long group = static_cast<long long>(kHostChunkBytes / p_head);
    if (group < 1) group = 1;
    if (group > bh) group = bh;
    for (int slot = 0; slot < 2; ++slot) {
        rc = staging_reserve(st, slot, 0, qk_head * group);
        if (rc == ATTNW_OK) rc = staging_reserve(st, slot, 1, qk_head * group);
        if (rc == ATTNW_OK) rc = staging_reserve(st, slot, 2, p_head * group);
        if (rc != ATTNW_OK) return rc;
    }
    const char* q = static_cast<const char*>(Q);
    const char* k = static_cast<const char*>(K);
    char* p = static_cast<char*>(P);
    int piece = 0;
    for (long long h0 = 0; h0 < bh; h0 += group, ++piece) {
        const long long g = (bh - h0 < group) ? bh - h0 : group;
        const int slot = piece & 1;
        cudaStream_t s = st->stream[slot];
        if (cudaMemcpyAsync(st->buf[slot][0], q + h0 * qk_head, g * qk_head, cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(st->buf[slot][1], k + h0 * qk_head, g * qk_head, cudaMemcpyHostToDevice, s) != cudaSuccess) {
            rc = ATTNW_ERR_CUDA;
            break;
        }
        rc = p_is_f32 ? attnw_fused_f32(st->buf[slot][0], st->buf[slot][1], st->buf[slot][2], 1, static_cast<int>(g), N,
                                        d, scale, s)
                      : attnw_fused(st->buf[slot][0], st->buf[slot][1], st->buf[slot][2], 1, static_cast<int>(g), N, d,
                                    scale, s);
        if (rc != ATTNW_OK) break;
        if (cudaMemcpyAsync(p + h0 * p_head, st->buf[slot][2], g * p_head, cudaMemcpyDeviceToHost, s) != cudaSuccess) {
            rc = ATTNW_ERR_CUDA;
            break;
        }
    }
    // On every path, also after an error: no copy may still be reading or writing the caller's buffers on return.
    for (int slot = 0; slot < 2; ++slot)
        if (cudaStreamSynchronize(st->stream[slot]) != cudaSuccess && rc == ATTNW_OK) rc = ATTNW_ERR_CUDA;
    if (rc != ATTNW_OK) return rc;
    return read_and_clear_status(nullptr);  // a wait that gave up inside a kernel: the result is not valid
}

int softmax_rows_host(const void* S, void* P, long long rows, long long cols, int p_is_f32) {
    const size_t esize = p_is_f32 ? 4 : 2;
    if (!S || !P) return ATTNW_ERR_NULL_POINTER;
    if (rows < 1 || cols < 1 || cols > (1ll << 40) || rows > (1ll << 40) || rows > (1ll << 62) / cols)
        return ATTNW_ERR_BAD_SHAPE;
    if (cols % 4 != 0) return ATTNW_ERR_MISALIGNED;
    HostStaging* st = nullptr;
    int rc = staging_for_current_device(&st);
    if (rc != ATTNW_OK) return rc;
    long long group = static_cast<long long>(kHostChunkBytes / (static_cast<unsigned long long>(cols) * 4ull));
    if (group < 1) group = 1;
    if (group > rows) group = rows;
    for (int slot = 0; slot < 2; ++slot) {
        rc = staging_reserve(st, slot, 0, static_cast<size_t>(group) * cols * 4);
        if (rc == ATTNW_OK) rc = staging_reserve(st, slot, 2, static_cast<size_t>(group) * cols * esize);
        if (rc != ATTNW_OK) return rc;
    }
    const char* src = static_cast<const char*>(S);
    char* dst = static_cast<char*>(P);
    int piece = 0;
    for (long long r0 = 0; r0 < rows; r0 += group, ++piece) {
        const long long g = (rows - r0 < group) ? rows - r0 : group;
        const int slot = piece & 1;
        cudaStream_t s = st->stream[slot];
        if (cudaMemcpyAsync(st->buf[slot][0], src + r0 * cols * 4, static_cast<size_t>(g) * cols * 4,
                            cudaMemcpyHostToDevice, s) != cudaSuccess) {
            rc = ATTNW_ERR_CUDA;
            break;
        }
        rc = p_is_f32 ? softmax_rows_f32(st->buf[slot][0], st->buf[slot][2], g, cols, s)
                      : softmax_rows(st->buf[slot][0], st->buf[slot][2], g, cols, s);
        if (rc != ATTNW_OK) break;
        if (cudaMemcpyAsync(dst + r0 * cols * esize, st->buf[slot][2], static_cast<size_t>(g) * cols * esize,
                            cudaMemcpyDeviceToHost, s) != cudaSuccess) {
            rc = ATTNW_ERR_CUDA;
            break;
        }
    }
    // On every path, also after an error: no copy may still be reading or writing the caller's buffers on return.
    for (int slot = 0; slot < 2; ++slot)
        if (cudaStreamSynchronize(st->stream[slot]) != cudaSuccess && rc == ATTNW_OK) rc = ATTNW_ERR_CUDA;
    if (rc != ATTNW_OK) return rc;
    return read_and_clear_status(nullptr);  // a wait that gave up inside a kernel: the result is not valid
}

int attnw_host_release(void) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ATTNW_ERR_CUDA;
    HostStaging& st = g_staging[dev];
    for (int slot = 0; slot < 2; ++slot) {
        if (st.streams_ready) cudaStreamSynchronize(st.stream[slot]);
        for (int w = 0; w < 3; ++w) {
            if (st.buf[slot][w]) cudaFree(st.buf[slot][w]);
            st.buf[slot][w] = nullptr;
            st.cap[slot][w] = 0;
        }
    }
    return ATTNW_OK;
}

int attnw_query_status(void* stream, unsigned int* device_status) {
    if (!device_status) return ATTNW_ERR_NULL_POINTER;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return ATTNW_ERR_CUDA;
    return read_and_clear_status(device_status);
}

int attnw_selftest_wait_timeout(long long limit_cycles, void* stream) {
    if (limit_cycles < 1 || limit_cycles > 2000000000ll) return ATTNW_ERR_BAD_SHAPE;  // at most about one second
    DeviceInfo* dev = nullptr;
    int rc = current_device(&dev);
    if (rc != ATTNW_OK) return rc;
    wait_timeout_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(limit_cycles);
    if (cudaGetLastError() != cudaSuccess) return ATTNW_ERR_CUDA;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return ATTNW_OK;
}

int attnw_selftest_exchange_tags(unsigned int next, void* stream) {
    DeviceInfo* dev = nullptr;
    int rc = current_device(&dev);
    if (rc != ATTNW_OK) return rc;
    unsigned long long id = 0;
    if (cudaStreamGetId(static_cast<cudaStream_t>(stream), &id) != cudaSuccess) {
        (void)cudaGetLastError();
        return ATTNW_ERR_CUDA;
    }
    GridrowAreas& areas = g_gridrow_areas[dev - g_devices];
    std::lock_guard<std::mutex> areas_lock(areas.mutex);
    uint32_t* tag = nullptr;
    for (int a = 0; a < areas.count && !tag; ++a)
        if (areas.area[a].stream_id == id) tag = &areas.area[a].tag;
    if (!tag) return ATTNW_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> noalloc_lock(g_mutex);
    uint32_t* noalloc_tag = &g_noalloc[dev - g_devices].tag;
    if (next > kLastTag || *tag > next || *noalloc_tag > next) return ATTNW_ERR_BAD_SHAPE;
    *tag = *noalloc_tag = next;
    return ATTNW_OK;
}

int attnw_set_fused_variant(int variant) {
    if (variant < 0 || variant > 4) return ATTNW_ERR_BAD_SHAPE;
    g_fused_variant.store(variant, std::memory_order_relaxed);
    return ATTNW_OK;
}

long long attnw_launch_count(int reset) {
    return reset ? g_launches.exchange(0, std::memory_order_relaxed) : g_launches.load(std::memory_order_relaxed);
}

const char* attnw_strerror(int code) {
    switch (code) {
        case ATTNW_OK: return "ok";
        case ATTNW_ERR_NULL_POINTER: return "a required pointer is NULL";
        case ATTNW_ERR_BAD_SHAPE: return "a size is out of range, or scale is negative or not finite";
        case ATTNW_ERR_MISALIGNED: return "a pointer or a row pitch is not a multiple of 16 bytes";
        case ATTNW_ERR_UNSUPPORTED: return "unsupported head dimension or device (needs d in {64,128}, sm_100)";
        case ATTNW_ERR_CUDA: return "a CUDA runtime or driver call failed";
        case ATTNW_ERR_TIMEOUT: return "a bounded device-side wait gave up; the output of that launch is undefined";
        case ATTNW_ERR_ALIASING: return "the output overlaps an input";
        default: return "unknown attnw status code";
    }
}

int attnw_version(void) { return kVersion; }
#ifdef ATTNW_TIMELINE
// Debug builds only (-DATTNW_TIMELINE=<cta index>): copies the cycle stamps of that CTA to the host.
int attnw_debug_timeline(long long* out) {
    if (cudaDeviceSynchronize() != cudaSuccess) return ATTNW_ERR_CUDA;
    return cudaMemcpyFromSymbol(out, attnw::g_attnw_timeline, sizeof(long long) * 32 * 160) == cudaSuccess ? ATTNW_OK
                                                                                                          : ATTNW_ERR_CUDA;
}
#endif

}  // extern "C"
