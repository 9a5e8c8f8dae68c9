// Queries and keys from the inputs for sm_100a: Q_h = X W^Q_h, K_h = X W^K_h for every head in one launch - the
// linear transformation in front of the attention weights (Section IV), which the paper leaves to the vendor's
// matmul and names as a step to bring into its own code (Section VIII).  The output is written head-major
// ([B, H, N, d], bf16), exactly what attnw_fused and attn_fused read, so no transposition pass is needed.
//
// A plain dense contraction, so it runs on the tensor cores, with the CTAs of a cluster of two as a pair (cta_group::2): a pair
// computes 256 rows of X times 256 output features (2 or 4 heads; Q's features, then K's), each CTA 128 of the rows and all of the
// features.  A CTA loads its rows and half of the features, so a byte of the operands in shared memory feeds twice the MMAs that it
// feeds within one CTA.  A pair stays for several tiles: tensor memory holds two accumulators, and 8 warps turn one into bf16 and store it
// while the tensor cores fill the other; the ring of 64-wide slices runs on from tile to tile.  launch_project chooses between whole
// tiles, a last round cut in two, and narrow tiles, by pairs or (small calls that pairs only hold up) by single CTAs.
// Weights are stored [H, d, d_model] (feature c of head h contiguous along d_model), which is the K-major B operand TMA can deliver as it is.
//
// What bounds it: large calls, the tensor pipe (512 cycles a slice) under the power cap; small ones, the latency of set-up, first load,
// epilogue and launch, some 5 us.  us per call, one CTA a tile of 256 x 256, 128 x 256 or 128 x 128 -> this kernel, B x N x d_model
// to H x d: 4 x 4096 x 4096 to 32 x 128 823 -> 724 .. 805 (by the box's power), 4 x 2825 x 1664 to 13 x 128 128 -> 106, 2 x 2092 x 368 to 37 x
// 64 28.6 -> 18.7, 1 x 2366 x 392 to 15 x 128 24.6 -> 13.5, 1 x 1000 x 1024 to 16 x 64 7.79 -> 6.66, 1 x 1757 x 768 to 12 x 64 8.17 -> 8.14; 547
// sizes, most of few tiles, together with the single CTAs 1.13 times as fast; behind: one head of 64 features, by 0.2 us (1 x 512 x 64 3.54 -> 3.75).
// What mattered in small calls: arrivals of the cluster's barrier and on the other CTA's mbarriers that order no memory (release costs
// about 1000 cycles each: 6.86 -> 5.33 us at 2 x 64 x 256 to 4 x 64); the divisions of the tile list in front of the set-up's waits, not
// of the first load (0.1 us); producers that a whole warp walks, with an elected lane, one for X and one for the weights (a lone lane took
// 475 cycles a slice, that warp alone 330, two 300).  Tiles of 512 x 256 or 256 x 512, with one accumulator: 1 to 14 % slower.
#pragma once
#include <cstddef>

#include "attnw_fused.cuh"

namespace attnw {
namespace proj {

constexpr int kKSlice = 64;          // d_model elements per stage: one 128-byte swizzle atom
constexpr int kRows = 128;           // rows of X of a CTA
constexpr int kFeatures = 128;       // features that a CTA loads for a whole tile (narrow tiles and halves: 64)
constexpr int kGroupTiles = 16;      // column tiles walked together (32 MB of weights at d_model = 4096)
constexpr int kEpiWarps = 8;         // TMEM lane quarter (4) x column half (2)
constexpr int kProducerX = 8;
constexpr int kMma = 9;
constexpr int kProducerW = 10;
constexpr int kThreads = 352;
constexpr int kAtomBytes = 128 * 128;           // 128 rows x 128 bytes
constexpr int kRingBytes = 192 * 1024;          // stages of [64-wide] slices: the rows of X, then the features
constexpr int kMaxStages = 6;
constexpr int kSlots = 2;                       // accumulators in tensor memory
constexpr int kSlotCols = kTmemCols / kSlots;
constexpr int kOutOff = kRingBytes;  // one staged store box per epilogue warp: 32 rows x 64 features
constexpr int kBarOff = kOutOff + kEpiWarps * kStageBoxBytes;
constexpr int kDynamicBytes = kBarOff + 256 + 1024;
static_assert(kDynamicBytes <= 227 * 1024, "shared memory budget");

enum : uint32_t {  // wait sites of this kernel (low byte of the status word)
    kSiteProducerEmpty = 112,
    kSiteMmaFull = 113,
    kSiteEpiAcc = 114,
    kSiteMmaAccEmpty = 115,
};

struct Barriers {
    uint64_t full[kMaxStages], empty[kMaxStages];    // full: the even CTA's, for both
    uint64_t acc_full[kSlots], acc_empty[kSlots];    // acc_empty: the even CTA's, for both
    uint32_t tmem_base;
    uint32_t abort_flag;
    uint32_t prior_failure;
    uint32_t peer_ran;  // written by the other CTA when it unwinds
    int loads;          // stages that a producer has asked for
};
static_assert(sizeof(Barriers) <= 256, "barrier block must fit its slot");

// The tiles of a call, the same arithmetic on the host and on the device.
struct Grid {
    int block;           // features that a CTA loads for a tile: kFeatures or half of that
    int feature_blocks;  // blocks of Q's features, and as many of K's behind them = column tiles (two blocks each)
    int row_blocks;      // blocks of kRows rows of a batch entry
    int row_tiles;       // of a row block for each CTA; they may belong to different batch entries
    __host__ __device__ Grid(int B, int N, int HD, int block_, int ctas)
        : block(block_), feature_blocks((HD - 1) / block_ + 1), row_blocks((N - 1) / kRows + 1), row_tiles((B * row_blocks + ctas - 1) / ctas) {}
    __host__ __device__ int tiles() const { return feature_blocks * row_tiles; }
};

// Whether the accumulator of item t is filled again by the same pair.  Only then does anyone wait for its release, and only then may the odd
// CTA send one: the even CTA might have ended before an arrival that nothing waits for.
__host__ __device__ constexpr bool accumulator_comes_again(int t, int pairs, int items) { return items - t > kSlots * pairs; }

// grid: clusters of two CTAs; pair p takes the items p, p + pairs, ...: the tiles 0 ... whole_tiles - 1, then the halves of the others.
// kPair = false: single CTAs, each in the place of a pair, with tiles of kRows rows and both blocks of features.
template <bool kPair>
__global__ void __launch_bounds__(kThreads, 1)
project_qk_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_wq,
                  const __grid_constant__ CUtensorMap tm_wk, const __grid_constant__ CUtensorMap tm_q,
                  const __grid_constant__ CUtensorMap tm_k, int B, int N, int d_model, int H, int d, int block, int whole_tiles) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Barriers* bars = reinterpret_cast<Barriers*>(smem + kBarOff);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    constexpr int kCtas = kPair ? 2 : 1;
    const int rank = kPair ? static_cast<int>(ptx::cluster_ctarank()) : 0;
    const Grid g(B, N, H * d, block, kCtas);
    const int items = 2 * g.tiles() - whole_tiles;
    const int first = static_cast<int>(blockIdx.x) / kCtas, pairs = static_cast<int>(gridDim.x) / kCtas;
    const int KT = (d_model + kKSlice - 1) / kKSlice;
    // The ring: six stages of one slice, or four of two narrow ones (single CTAs, with all features: four and three): a stage costs each of the
    // issuing warps some 300 cycles, which the 256 of the MMAs of one narrow slice do not cover (1 x 512 x 4096 to 8 x 128 14.6 -> 13.3 us).
    const int slice_bytes = kAtomBytes + (kPair ? block : 2 * block) * 128;
    const int slices = block == kFeatures ? 1 : 2;
    const int stage_bytes = slices * slice_bytes;
    const int stages = kPair ? (block == kFeatures ? kMaxStages : 4) : (block == kFeatures ? 4 : 3);  // kRingBytes of them
    // The ring's stages in turn, and how often a stage has been used before, modulo 2.
    struct Turn {
        int s = 0;
        uint32_t parity = 0;
        __device__ __forceinline__ void next(int stages) {
            if (++s == stages) {
                s = 0;
                parity ^= 1u;
            }
        }
    };
    // Column tiles are walked in groups: within a group the tiles of one block of rows are neighbours (that block of X is fetched once
    // per group), and the group's slice of the weights is small enough to stay in L2 while all row blocks pass.
    struct Item {
        int block;    // the column tile's first block of features, of Q's, then of K's
        int half;     // of the blocks; -1 = both halves
        int row_tile;
        int b, row;   // this CTA's rows: batch entry (B = none) and first row
    };
    auto item = [&](int t) {
        Item r;
        r.half = t < whole_tiles ? -1 : (t - whole_tiles) & 1;
        if (t >= whole_tiles) t = whole_tiles + ((t - whole_tiles) >> 1);
        const int groups = (g.feature_blocks + kGroupTiles - 1) / kGroupTiles;
        const int group = groups == 1 ? 0 : min(t / (kGroupTiles * g.row_tiles), groups - 1);
        const int in_group = t - group * kGroupTiles * g.row_tiles;
        const int width = group == groups - 1 ? g.feature_blocks - group * kGroupTiles : kGroupTiles;
        r.row_tile = in_group / width;
        r.block = 2 * (group * kGroupTiles + in_group - r.row_tile * width);
        const int rb = kCtas * r.row_tile + rank;
        r.b = rb / g.row_blocks;
        r.row = (rb - r.b * g.row_blocks) * kRows;
        return r;
    };
    // (the first one here: the divisions run beside the set-up, and not in front of the first load)
    const Item first_item = item(first);

    // ---- set-up ------------------------------------------------------------------------------
    if (threadIdx.x == 0) {
        ptx::grid_dependency_wait();
        const uint32_t prior_failure = *reinterpret_cast<volatile unsigned int*>(&g_attnw_status);  // (arrives meanwhile)
        for (int s = 0; s < stages; ++s) {
            ptx::mbar_init(&bars->full[s], 1);
            ptx::mbar_init(&bars->empty[s], 1);
        }
        for (int s = 0; s < kSlots; ++s) {
            ptx::mbar_init(&bars->acc_full[s], 1);
            ptx::mbar_init(&bars->acc_empty[s], kCtas * kEpiWarps);
        }
        bars->abort_flag = prior_failure;
        bars->peer_ran = 0;
        bars->loads = 0;
        bars->prior_failure = prior_failure;
        ptx::mbar_fence_init();
    }
    if (warp == kProducerX && lane == 0) {
        ptx::prefetch_tensormap(&tm_x);
        ptx::prefetch_tensormap(&tm_wq);
        ptx::prefetch_tensormap(&tm_wk);
        ptx::prefetch_tensormap(&tm_q);
        ptx::prefetch_tensormap(&tm_k);
    }
    if (warp == kMma) {
        if constexpr (kPair) {
            ptx::pair_tmem_alloc(&bars->tmem_base, kTmemCols);
            ptx::pair_tmem_relinquish();
        } else {
            ptx::tmem_alloc(&bars->tmem_base, kTmemCols);
            ptx::tmem_relinquish();
        }
    }
    ptx::grid_dependency_wait();
    ptx::tc_fence_before_sync();
    __syncthreads();
    if constexpr (kPair) {
        ptx::cluster_arrive_relaxed();
        ptx::cluster_wait_acquire();
    }
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    // An earlier launch gave up: do not queue more waits behind it.  Should the word be cleared between the two CTAs' looks at it, the one that
    // has seen it tells the other in the teardown, where nothing is stored yet: each tile needs both CTAs' loads and the even one's MMAs.
    const bool run = bars->prior_failure == 0u;

    if (run && (warp == kProducerX || warp == kProducerW)) {
        // ================= TMA producers, of rows and of features: per stage a 64-wide slice =================
        const bool for_rows = warp == kProducerX;
        const uint64_t keep = ptx::policy_evict_last();
        const uint32_t empty0 = ptx::smem_u32(&bars->empty[0]);
        const uint32_t full0 = kPair ? ptx::map_to_cta(ptx::smem_u32(&bars->full[0]), 0) : ptx::smem_u32(&bars->full[0]);
        bool ok = true;
        Turn turn;
        int n = 0;  // stages asked for
        Item it = first_item;
        for (int t = first; ok && t < items;) {
            const int block = it.block + rank;
            const bool keys = block >= g.feature_blocks;
            const bool wide = kPair && it.half < 0 && g.block == kFeatures;
            const CUtensorMap* map = for_rows ? &tm_x : keys ? &tm_wk : &tm_wq;
            // a single CTA loads the column tile's second block too
            const bool keys2 = it.block + 1 >= g.feature_blocks;
            const int c1_2 = (keys2 ? it.block + 1 - g.feature_blocks : it.block + 1) * g.block;
            const int c1 = for_rows ? it.row : (keys ? block - g.feature_blocks : block) * g.block + (it.half == 1 ? kFeatures / 2 : 0);
            const int c2 = for_rows ? it.b : 0;
            // An odd number of row blocks leaves a CTA without rows: what its MMAs make of old contents is never stored.
            const bool load = !for_rows || it.b < B;
            const uint32_t bytes = !kPair ? static_cast<uint32_t>(slice_bytes)
                                          : static_cast<uint32_t>((2 * it.row_tile + 1 < B * g.row_blocks ? 2 : 1) + (wide ? 2 : 1)) * kAtomBytes;  // of both CTAs
            for (int kt = 0; kt < KT; kt += slices, ++n, turn.next(stages)) {
                ok = warp_wait(empty0 + 8u * static_cast<uint32_t>(turn.s), turn.parity ^ 1u, abort_flag, kSiteProducerEmpty);
                if (!ok) break;
                uint8_t* st = smem + turn.s * stage_bytes + (for_rows ? 0 : kAtomBytes);
                const uint32_t full = full0 + 8u * static_cast<uint32_t>(turn.s);
                const bool second = slices == 2 && kt + 1 < KT;
                if (ptx::elect_one()) {
                    if (rank == 0 && for_rows) ptx::mbar_expect_tx(&bars->full[turn.s], second ? 2 * bytes : bytes);
                    // rows or features beyond the tensor's extent, and d_model's ragged tail, arrive as zeros
                    if constexpr (kPair) {
                        if (load) ptx::pair_tma_load_3d(st, map, full, kt * kKSlice, c1, c2, keep);
                        if (load && second) ptx::pair_tma_load_3d(st + slice_bytes, map, full, (kt + 1) * kKSlice, c1, c2, keep);
                        if (wide && !for_rows) ptx::pair_tma_load_3d(st + kAtomBytes / 2, map, full, kt * kKSlice, c1 + kFeatures / 2, c2, keep);
                    } else {
                        for (int i = 0; i < (second ? 2 : 1); ++i) {
                            uint8_t* to = st + i * slice_bytes;
                            const int c0 = (kt + i) * kKSlice;
                            if (for_rows) {
                                ptx::tma_load_3d(to, map, &bars->full[turn.s], c0, c1, c2, keep);
                            } else {
                                for (int f = 0; f < g.block; f += kFeatures / 2) {
                                    ptx::tma_load_3d(to + f * 128, map, &bars->full[turn.s], c0, c1 + f, 0, keep);
                                    ptx::tma_load_3d(to + (g.block + f) * 128, keys2 ? &tm_wk : &tm_wq, &bars->full[turn.s], c0, c1_2 + f, 0, keep);
                                }
                            }
                        }
                    }
                }
                __syncwarp();
            }
            t += pairs;
            if (t < items) it = item(t);
        }
        if (lane == 0) atomicMax(&bars->loads, n);
        // The MMAs' arrivals on this CTA's barriers are all here before it ends.
        for (int i = n > stages ? n - stages : 0; ok && i < n; ++i)
            ok = warp_wait(empty0 + 8u * static_cast<uint32_t>(i % stages), static_cast<uint32_t>(i / stages) & 1u, abort_flag, kSiteProducerEmpty);
    } else if (run && warp == kMma && rank == 0) {
        // ================= MMA issuer, for both CTAs =================
        constexpr uint32_t idesc_whole = ptx::umma_idesc_bf16_f32(kCtas * kRows, 2 * kFeatures);
        constexpr uint32_t idesc_half = ptx::umma_idesc_bf16_f32(kCtas * kRows, kFeatures);
        auto mma = [](uint32_t to, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
            if constexpr (kPair)
                ptx::pair_umma_f16_ss(to, a, b, idesc, accumulate);
            else
                ptx::umma_f16_ss(to, a, b, idesc, accumulate);
        };
        auto commit = [](uint64_t* bar) {
            if constexpr (kPair)
                ptx::pair_umma_commit(bar);
            else
                ptx::umma_commit(bar);
        };
        const uint64_t base = ptx::umma_desc_kmajor_sw128(ptx::smem_u32(smem));
        bool ok = true;
        const uint32_t full0 = ptx::smem_u32(&bars->full[0]);
        uint64_t st = base;  // of the stage that is next
        Turn turn;
        int use = 0;  // accumulators begun
        for (int t = first; ok && t < items; t += pairs, ++use) {
            const uint32_t idesc = t < whole_tiles && block == kFeatures ? idesc_whole : idesc_half;
            const int slot = use % kSlots;
            ok = warp_wait(ptx::smem_u32(&bars->acc_empty[slot]), (static_cast<uint32_t>(use / kSlots) & 1u) ^ 1u, abort_flag, kSiteMmaAccEmpty);
            ptx::tc_fence_after_sync();
            const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(slot * kSlotCols);
            for (int kt = 0; ok && kt < KT; kt += slices) {
                ok = warp_wait(full0 + 8u * static_cast<uint32_t>(turn.s), turn.parity, abort_flag, kSiteMmaFull);
                if (!ok) break;
                if (ptx::elect_one()) {
#pragma unroll
                    for (int k = 0; k < kKSlice / 16; ++k)
                        mma(d_tmem, st + static_cast<uint64_t>((k * 32) >> 4), st + static_cast<uint64_t>((kAtomBytes + k * 32) >> 4), idesc,
                            (kt > 0 || k > 0) ? 1u : 0u);
                    if (slices == 2 && kt + 1 < KT) {
                        const uint64_t second = st + static_cast<uint64_t>(slice_bytes >> 4);
#pragma unroll
                        for (int k = 0; k < kKSlice / 16; ++k)
                            mma(d_tmem, second + static_cast<uint64_t>((k * 32) >> 4), second + static_cast<uint64_t>((kAtomBytes + k * 32) >> 4), idesc, 1u);
                    }
                    commit(&bars->empty[turn.s]);
                    if (kt + slices >= KT) commit(&bars->acc_full[slot]);
                }
                __syncwarp();
                st += static_cast<uint64_t>(stage_bytes >> 4);
                turn.next(stages);
                if (turn.s == 0) st = base;
            }
        }
    } else if (run && warp < kEpiWarps) {
        // ================= Epilogue warps: accumulators -> bf16 -> shared memory -> TMA stores, head-major =================
        const int quarter = warp & 3;
        const int ch = warp >> 2;  // this warp takes the columns of the item's block `ch` of features (a pair: those that CTA `ch` has loaded)
        const uint32_t sw = static_cast<uint32_t>(lane & 7);
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t own_box = ptx::smem_u32(smem + kOutOff + warp * kStageBoxBytes), ring_box = ptx::smem_u32(smem + warp * kStageBoxBytes);
        const uint64_t keep = ptx::policy_evict_last();  // the attention kernels read Q and K next
        bool ok = true;
        int use = 0;
        Item it = first_item;
        for (int t = first; ok && t < items; ++use) {
            const int row = it.row + quarter * 32;
            const bool rows_exist = it.b < B && row < N;
            const int block = it.block + ch;
            const bool keys = block >= g.feature_blocks;
            const int width = it.half < 0 ? g.block : kFeatures / 2;
            const int c0 = (keys ? block - g.feature_blocks : block) * g.block + (it.half == 1 ? kFeatures / 2 : 0);
            int head = d == 64 ? c0 >> 6 : c0 >> 7, offset = c0 & (d - 1);  // of the box's first feature
            const bool last = t + pairs >= items;
            const int slot = use % kSlots;
            const uint32_t taddr = t_lane + static_cast<uint32_t>(slot * kSlotCols + ch * width);
            ok = warp_wait(ptx::smem_u32(&bars->acc_full[slot]), static_cast<uint32_t>(use / kSlots) & 1u, abort_flag, kSiteEpiAcc);
            if (!ok) break;
            ptx::tc_fence_after_sync();
#pragma unroll 1
            for (int c = 0; c < width; c += 64) {
                uint32_t v[2][32];
                ptx::tmem_ld_32x32b_x32(taddr + static_cast<uint32_t>(c), v[0]);
                ptx::tmem_ld_32x32b_x32(taddr + static_cast<uint32_t>(c + 32), v[1]);
                ptx::tmem_wait_ld();
                if (c + 64 == width && accumulator_comes_again(t, pairs, items)) {  // it may be overwritten
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (kPair)
                            ptx::mbar_arrive_cluster_relaxed(ptx::map_to_cta(ptx::smem_u32(&bars->acc_empty[slot]), 0));
                        else
                            ptx::mbar_arrive(&bars->acc_empty[slot]);
                    }
                }
                // The box: once the store that used it last has read it (lane 0 has issued them all).  The last tile's second one has room
                // of its own, in the ring, which nothing uses any more.
                const uint32_t box = last && c > 0 ? ring_box : own_box;
                if (box == own_box) ptx::bulk_wait_group_read<0>();
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {  // one 16-byte piece of the row's 128 bytes
                    uint32_t w[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        w[j] = ptx::pack_bf16x2(__uint_as_float(v[i >> 2][(i & 3) * 8 + 2 * j]), __uint_as_float(v[i >> 2][(i & 3) * 8 + 2 * j + 1]));
                    ptx::st_shared_v4(box + static_cast<uint32_t>(lane * 128) + ((static_cast<uint32_t>(i) ^ sw) << 4), w[0], w[1], w[2], w[3]);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && rows_exist && head < H) {
                    ptx::tma_store_3d(keys ? &tm_k : &tm_q, box, offset, row, it.b * H + head, keep);
                    ptx::bulk_commit_group();
                }
                offset += 64;
                if (offset == d) {
                    offset = 0;
                    ++head;
                }
            }
            t += pairs;
            if (t < items) it = item(t);
        }
        ptx::bulk_wait_group<0>();
    }

    // ---- teardown: every role of both CTAs falls through to here, also after a wait gave up ----
    ptx::tc_fence_before_sync();
    __syncthreads();
    if constexpr (kPair) {
        if (threadIdx.x == 0 && *abort_flag) {
            ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&bars->abort_flag), rank ^ 1), 1u);
            if (run) ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&bars->peer_ran), rank ^ 1), 1u);
            ptx::fence_cluster();
        }
        __syncwarp();
        ptx::cluster_arrive_relaxed();
        ptx::cluster_wait_acquire();
    }
    ptx::tc_fence_after_sync();
    if (*abort_flag) {
        // Unwinding: let the MMAs of the pair and the arrivals on either CTA that nobody has waited for come to their end, and the copies of both
        // CTAs land, before shared and tensor memory are released.
        if (run || bars->peer_ran) wait_for_late_stores();
        if (rank == 0 && threadIdx.x == 0) {
            const int mine = bars->loads;
            const int theirs = kPair ? static_cast<int>(ptx::ld_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&bars->loads), 1))) : 0;
            const int last = mine > theirs ? mine : theirs;
            const long long t0 = clock64();
            // (the phase of a stage that only one of the producers has asked for does not end: there the limit runs out)
            for (int i = last > stages ? last - stages : 0; i < last; ++i)
                while (!ptx::mbar_try_wait(&bars->full[i % stages], static_cast<uint32_t>(i / stages) & 1u) &&
                       clock64() - t0 < kWaitLimitCycles / 8) {
                }
        }
        __syncwarp();
        if constexpr (kPair) {
            ptx::cluster_arrive_relaxed();
            ptx::cluster_wait_acquire();
        } else {
            __syncthreads();
        }
    }
    if (warp == kMma) {
        if constexpr (kPair)
            ptx::pair_tmem_dealloc(tmem_base, kTmemCols);
        else
            ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

}  // namespace proj
}  // namespace attnw
