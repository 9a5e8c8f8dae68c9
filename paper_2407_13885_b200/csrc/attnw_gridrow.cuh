// Grid-row fused attention-weight kernel for sm_100a: the SRAM-resident design of Section VII of the paper
// with the roles of a Tensix grid row taken by a GROUP of CTAs that the kernel forms itself.
//
// The paper lays the score matrix out over a grid of cores; the cores of one grid row hold the pieces of the
// same rows of scores, compute LOCAL row maxima and sums and exchange them to obtain the GLOBAL ones before
// normalising (Section VII; Eq. 1).  Here a group of C = ceil(N / 256) CTAs owns a 128-row block of one head; CTA r
// of the group works on the 128 x 256 slab of scores for keys [256 r, 256 r + 256).  Tensor cores and exponentials
// run once per element.
//
// Tensor memory, bfloat16 output:
//   columns [0, 128)    the landing slot: the MMA writes float32 scores of 128 keys here; it goes back to the MMA issuer
//                       as soon as its scores are in registers
//   columns [128, 512)  three packed regions, used by the row blocks in turn: the exponentials as f16 pairs, waiting
//                       for the row's statistics
// so two further row blocks can be computed, and their exponentials taken, while the statistics of one cross the
// group.  (f16 keeps 11 bits of e in [0, 1]: 5e-4 relative, next to the 2e-3 of the bf16 result.)
// Tensor memory, float32 output: two regions of 256 columns; the exponentials replace the scores as float32, and a slot of
// 128 columns goes back to the MMA issuer when its weights have been staged.
//
// Groups are not hardware clusters (clusters of 8 or 16 CTAs cannot occupy every SM): the grid is launched
// cooperatively with one CTA per SM, consecutive CTAs form a group, and the 16-byte (offset, sum) pair of a row
// travels through L2 as two 8-byte words that each carry a tag {value, tag, value, tag}; a reader accepts a
// pair once both tags name the row block it is waiting for.  No fence, no flag, no atomics: the tag arrives
// with the value in one 8-byte store.  Every poll is bounded.
//   C = 1          no exchange: the pair stays in shared memory
//   2 <= C <= 4    every CTA reads the C pairs of each row and reduces them redundantly, as the paper's kernel does
//   C > 4          the rows of a block are dealt out to the CTAs; a row's owner reads its C pairs, reduces them once and
//                  posts (M, 1/L) for all (the exchange of Section VIII).  One more hop through L2, but two loads per row
//                  and CTA instead of C, and C may be larger than 16.
//
// Roles of a CTA (896 threads, 28 warps; warp w may touch TMEM lanes 32 (w % 4) ...):
//   warps 0-15   exponentials, all sixteen on ONE row block at a time: four threads per row, thread (row, g) takes columns
//                [32 g, 32 g + 32) of both slots: scores to registers, maximum, offset mb, e = 2^(c s - mb), sum, e back
//                to tensor memory; the thread's (mb, l) to shared memory; the last of a row's four warps to finish
//                merges the parts and posts the row's pair
//   warps 16-19  normalise the even row blocks (20-23: the odd ones): a thread owns one row; takes the row's M and 1/L,
//                then per box of 128 bytes a row p = e * 2^(mb - M) / L, rounded to the output type, staged and stored by
//                one TMA store per warp (32 rows x 128 bytes) and box; P is written exactly once
//   warp 24      TMA producer: the CTA's key slab once per head (it stays in shared memory while the group walks
//                the head's row blocks), one query tile per row block
//   warp 25      tcgen05.mma issuer (one elected lane)
//   warps 26-27  the owner's reduction of the row block, half of its rows each
//
// With -DATTNW_TIMELINE=<CTA> one lane per role of that CTA stamps clock64() per row block (events, by index):
//   13 MMA of the block issued | 0 exponentials begin, 2 slot 0 ready, 17/20 load of slot k, 16/19 maximum known,
//   18/21 exponentials of slot k done, 24/26 e stored, 4 parts posted | 22 owner begins to wait, 23 pairs seen,
//   25 result posted | 10 normalise begins to wait, 6 own CTA done, 11 statistics seen, 12 box 0 read,
//   14/15/8/9 box 2 read / staging free / staged / stored, 7 block done.
#pragma once
#include "attnw_resident.cuh"

namespace attnw {
namespace gr {

constexpr int kSlabCols = 256;                       // key columns per CTA and row block
constexpr int kSub = 128;                            // columns per MMA slot
constexpr int kSubsPerBlock = kSlabCols / kSub;
constexpr int kPackedCol0 = kSub;                    // packed exponentials: columns [128, 512), 128 per region
constexpr int kPackedCols = kSlabCols / 2;           // two f16 per 32-bit column
constexpr int kChunksPerBlock = kSlabCols / kChunk;  // 32-column chunks, each with its own offset
constexpr int kExpWarps = 16;
constexpr int kParts = kExpWarps / 4;                // threads per row
constexpr int kNormWarp0 = kExpWarps;
constexpr int kProducerWarpG = kNormWarp0 + 8;
constexpr int kMmaWarpG = kProducerWarpG + 1;
constexpr int kOwnerWarpG = kProducerWarpG + 2;
constexpr int kThreads = 32 * (kOwnerWarpG + 2);
constexpr int kStageBytes = 32 * 128;                // one staged store box: 32 rows x 128 bytes
constexpr int kMaxDirectCtas = 4;                    // up to here every CTA reads all pairs of a row
constexpr int kMaxGroupCtas = 128;
constexpr int kMaxN = 4096;                          // what variant 4 and attnw_fused_noalloc serve
constexpr int kXchgDepth = 8;    // row blocks i and i + 8 of a group share exchange entries (see the proof at the owner)

enum : uint32_t {  // wait sites of this kernel (low byte of the status word)
    kSiteGrKEmpty = 32,
    kSiteGrQEmpty = 33,
    kSiteGrQFull = 34,
    kSiteGrKFull = 35,
    kSiteGrSlotFree = 36,
    kSiteGrSFull = 37,
    kSiteGrPosted = 38,
    kSiteGrExchange = 39,
    kSiteGrOwner = 42,
};

template <int D>
struct Smem {
    static constexpr int kQStages = 2;  // query tiles in shared memory (with one, the load of the next tile shows: 1.28 against 1.13 ms)
    static constexpr int kStages = (D == 128) ? 2 : 4;  // staged boxes per normalise warp
    static constexpr int kAtoms = D / 64;
    static constexpr int kAtomBytes = kTile * 128;
    static constexpr int kTileBytes = kAtoms * kAtomBytes;
    static constexpr int kKAtomBytes = kSlabCols * 128;                 // key slab, atom-major: [d / 64][256 keys][128 bytes]
    static constexpr int kKOff = 0;
    static constexpr int kQOff = kKOff + 2 * kTileBytes;
    static constexpr int kOutOff = kQOff + kQStages * kTileBytes;       // staging boxes [8 warps][kStages]
    static constexpr int kMbcOff = kOutOff + 8 * kStages * kStageBytes; // float mbc[3 regions][8 chunks][128 rows]: offset per chunk
    static constexpr int kPartOff = kMbcOff + 3 * kChunksPerBlock * kTile * 4;  // float2 part[3 regions][4][128 rows]
    static constexpr int kBarOff = kPartOff + 3 * kParts * kTile * 8;
    static constexpr int kBytes = kBarOff + 512;
    static constexpr int kDynamicBytes = kBytes + 1024;
};
static_assert(Smem<128>::kDynamicBytes <= 227 * 1024 && Smem<64>::kDynamicBytes <= 227 * 1024, "shared memory budget");

struct Barriers {
    uint64_t k_full, k_empty;
    uint64_t q_full[2], q_empty[2];
    uint64_t s_full[2 * kSubsPerBlock], s_free[2 * kSubsPerBlock];  // slots: scores ready / slot may be overwritten
    uint64_t pk_free[3][kSlabCols / 64];                    // [region][64 columns]: the packed exponentials have been read
    uint64_t posted[3];
    uint32_t parts_done[3][4];   // [region][TMEM lane quarter]: exponential warps that have finished a row's parts (never reset)
    uint32_t tmem_base;
    uint32_t abort_flag;
    uint32_t prior_failure;
};
static_assert(sizeof(Barriers) <= 512, "barrier block must fit its slot");

__device__ __forceinline__ void st_message(uint4* p, float a, float b, uint32_t tag) {
    asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(__float_as_uint(a)), "r"(tag),
                 "r"(__float_as_uint(b)), "r"(tag)
                 : "memory");
}
__device__ __forceinline__ uint4 ld_message(const uint4* p) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

// Loads `n` <= K messages until all of them carry `tag` for every lane of the warp (entries beyond n repeat the last).
// false = the time limit ran out, or another role gave up.
template <int K, typename Addr>
__device__ __forceinline__ bool poll_messages(uint4 (&v)[K], int n, uint32_t tag, volatile uint32_t* abort_flag, uint32_t site, Addr addr) {
    const long long t0 = clock64();
    for (uint32_t spin = 1;; ++spin) {
        // all loads first, then the tags: one round trip to L2 a round
#pragma unroll
        for (int c = 0; c < K; ++c) v[c] = ld_message(addr(c < n ? c : n - 1));
        bool valid = true;
#pragma unroll
        for (int c = 0; c < K; ++c) valid = valid && v[c].y == tag && v[c].w == tag;
        if (__all_sync(0xffffffffu, valid)) return true;
        if ((spin & 15u) == 0) {
            bool give_up = *abort_flag != 0u;
            if (!give_up && clock64() - t0 > kWaitLimitCycles) {
                *abort_flag = 1;
                atomicCAS(&g_attnw_status, 0u, 0x80000000u | site);
                give_up = true;
            }
            if (__any_sync(0xffffffffu, give_up)) return false;
        }
    }
}

// The first CTAs of a group of C > kMaxDirectCtas own the rows of a block: a power of two of them, 128 / that many rows each.
__host__ __device__ constexpr int owner_count(int group_ctas) {
    int n = 4;
    while (2 * n <= group_ctas && 2 * n <= kTile) n *= 2;
    return n;
}

// xchg: [grid CTAs][kXchgDepth][128 rows] pairs, then [groups][kXchgDepth][128 rows] results, messages of 16 bytes in
// memory owned by the library, zero before first use.
// tag_base: tags tag_base + 1 ... tag_base + (row blocks of the longest list) belong to this launch alone.
template <int D, typename OutT>
__global__ void __launch_bounds__(kThreads, 1)
attnw_gridrow_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_p, int N, int total_items, int group_ctas, int n_groups,
                     float scale_log2e, uint4* __restrict__ xchg, uint32_t tag_base) {
    using L = Smem<D>;
    constexpr bool kF32 = sizeof(OutT) == 4;
    constexpr int kBoxCols = 128 / sizeof(OutT);  // columns of one staged store box
    constexpr int kMaxBoxes = kSlabCols / kBoxCols;
    constexpr int kRegions = kF32 ? 2 : 3;        // row blocks whose exponentials tensor memory holds
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Barriers* bars = reinterpret_cast<Barriers*>(smem + L::kBarOff);
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int group = static_cast<int>(blockIdx.x) / group_ctas;
    const int rank = static_cast<int>(blockIdx.x) % group_ctas;
    if (group >= n_groups) return;  // CTAs beyond the last whole group have no part in the launch
    const int T = (N + kTile - 1) / kTile;                          // row blocks per head
    const int col0 = rank * kSlabCols;                              // first key of this CTA's slab
    const int width = (N - col0 < kSlabCols) ? N - col0 : kSlabCols;  // keys of the slab that exist (>= 1)
    const int n_sub = (width + kSub - 1) / kSub;                    // MMA slots in use = 128-key tiles of the slab, 1..2
    const int n_boxes = (width + kBoxCols - 1) / kBoxCols;          // store boxes in use
    // The group's list: a contiguous range of (head, row block) items, so that the key slab changes rarely.
    const long long begin_ll = static_cast<long long>(total_items) * group / n_groups;
    const long long end_ll = static_cast<long long>(total_items) * (group + 1) / n_groups;
    const int begin = static_cast<int>(begin_ll);
    const int n_items = static_cast<int>(end_ll - begin_ll);
    uint4* const results = xchg + (static_cast<size_t>(n_groups) * group_ctas + group) * kXchgDepth * kTile;

    // ---- set-up ------------------------------------------------------------------------------
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bars->k_full, 1);
        ptx::mbar_init(&bars->k_empty, 1);
        for (int j = 0; j < 2 * kSubsPerBlock; ++j) {
            ptx::mbar_init(&bars->s_full[j], 1);
            ptx::mbar_init(&bars->s_free[j], kF32 ? 4 : kExpWarps);  // one arrival per warp that reads the slot last
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(&bars->q_full[s], 1);
            ptx::mbar_init(&bars->q_empty[s], 1);
        }
        for (int r = 0; r < 3; ++r) {
            for (int b = 0; b < kSlabCols / 64; ++b) ptx::mbar_init(&bars->pk_free[r][b], 4);  // the row block's normalise warps
            ptx::mbar_init(&bars->posted[r], kExpWarps);
            for (int x = 0; x < 4; ++x) bars->parts_done[r][x] = 0;
        }
        bars->abort_flag = 0;
        bars->prior_failure = *reinterpret_cast<volatile unsigned int*>(&g_attnw_status);
        ptx::mbar_fence_init();
    }
    if (warp == kProducerWarpG && lane == 0) {
        ptx::prefetch_tensormap(&tm_q);
        ptx::prefetch_tensormap(&tm_k);
        ptx::prefetch_tensormap(&tm_p);
    }
    if (warp == kMmaWarpG) {
        ptx::tmem_alloc(&bars->tmem_base, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    const bool run = bars->prior_failure == 0u && n_items > 0;  // an earlier launch step gave up: skip the work

    // Slots.  bfloat16: one for all; float32: two per region.
    auto slot_of = [](int i, int j) { return kF32 ? (i & 1) * kSubsPerBlock + j : 0; };
    auto slot_use = [n_sub](int i, int j) { return static_cast<uint32_t>(kF32 ? i >> 1 : i * n_sub + j); };  // how often the slot has been used before

    if (run && warp == kProducerWarpG) {
        // ================= TMA producer =================
        if (lane == 0) {
            const uint64_t keep = ptx::policy_evict_last();
            int cur_bh = -1;
            uint32_t heads = 0;
            int issued = 0;
            for (int i = 0; i < n_items; ++i) {
                const int gi = begin + i, bh = gi / T, rb = gi % T;
                if (bh != cur_bh) {  // new head: the slab may be replaced once every MMA of the old head has read it
                    if (!fused_wait(&bars->k_empty, (heads & 1u) ^ 1u, abort_flag, kSiteGrKEmpty)) break;
                    ptx::mbar_expect_tx(&bars->k_full, static_cast<uint32_t>(n_sub * L::kTileBytes));
                    for (int t = 0; t < n_sub; ++t)
                        for (int a = 0; a < L::kAtoms; ++a)
                            ptx::tma_load_3d(smem + L::kKOff + a * L::kKAtomBytes + t * L::kAtomBytes, &tm_k, &bars->k_full,
                                             a * 64, col0 + t * kTile, bh, keep);
                    ++heads;
                    cur_bh = bh;
                }
                const int qs = i % L::kQStages;
                const uint32_t uq = static_cast<uint32_t>(i / L::kQStages);
                if (!fused_wait(&bars->q_empty[qs], (uq & 1u) ^ 1u, abort_flag, kSiteGrQEmpty)) break;
                ptx::mbar_expect_tx(&bars->q_full[qs], static_cast<uint32_t>(L::kTileBytes));
                for (int a = 0; a < L::kAtoms; ++a)
                    ptx::tma_load_3d(smem + L::kQOff + qs * L::kTileBytes + a * L::kAtomBytes, &tm_q, &bars->q_full[qs], a * 64,
                                     rb * kTile, bh, keep);
                issued = i + 1;
            }
            if (*abort_flag) {
                // Unwinding: let the copies already in flight land before shared memory is released.
                const long long t0 = clock64();
                if (heads > 0)
                    while (!ptx::mbar_try_wait(&bars->k_full, (heads - 1u) & 1u) && clock64() - t0 < kWaitLimitCycles / 8) {
                    }
                for (int back = 1; back <= 2 && back <= issued; ++back) {
                    const int i = issued - back;
                    while (!ptx::mbar_try_wait(&bars->q_full[i % L::kQStages], static_cast<uint32_t>(i / L::kQStages) & 1u) &&
                           clock64() - t0 < kWaitLimitCycles / 4) {
                    }
                }
            }
        }
    } else if (run && warp == kMmaWarpG) {
        // ================= MMA issuer (warp-uniform loop, one elected lane issues) =================
        constexpr uint32_t idesc = ptx::umma_idesc_bf16_f32(kTile, kSub);
        const uint32_t q_addr = ptx::smem_u32(smem + L::kQOff);
        const uint32_t k_addr = ptx::smem_u32(smem + L::kKOff);
        int cur_bh = -1;
        uint32_t heads = 0;
        bool ok = true;
        for (int i = 0; ok && i < n_items; ++i) {
            const int gi = begin + i, bh = gi / T;
            const int qs = i % L::kQStages;
            ok = __all_sync(0xffffffffu, fused_wait(&bars->q_full[qs], static_cast<uint32_t>(i / L::kQStages) & 1u, abort_flag, kSiteGrQFull));
            if (!ok) break;
            if (bh != cur_bh) {
                ok = __all_sync(0xffffffffu, fused_wait(&bars->k_full, heads & 1u, abort_flag, kSiteGrKFull));
                if (!ok) break;
                ++heads;
                cur_bh = bh;
            }
            const bool last_of_head = (i + 1 == n_items) || ((gi + 1) / T != bh);
            for (int j = 0; ok && j < n_sub; ++j) {
                const int slot = slot_of(i, j);
                ok = __all_sync(0xffffffffu, fused_wait(&bars->s_free[slot], (slot_use(i, j) & 1u) ^ 1u, abort_flag, kSiteGrSlotFree));
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (lane == 0 && j == 0) ATTNW_STAMP(13, i);
                const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(slot * kSub);
                const uint32_t a_addr = q_addr + static_cast<uint32_t>(qs * L::kTileBytes);
                const uint32_t b_addr = k_addr + static_cast<uint32_t>(j * kSub * 128);  // keys kSub j ... of every atom
                if (ptx::elect_one()) {
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) {
                        const uint32_t a_off = static_cast<uint32_t>((k >> 2) * L::kAtomBytes + (k & 3) * 32);
                        const uint32_t b_off = static_cast<uint32_t>((k >> 2) * L::kKAtomBytes + (k & 3) * 32);
                        ptx::umma_f16_ss(d_tmem, ptx::umma_desc_kmajor_sw128(a_addr + a_off),
                                         ptx::umma_desc_kmajor_sw128(b_addr + b_off), idesc, k > 0 ? 1u : 0u);
                    }
                    ptx::umma_commit(&bars->s_full[slot]);
                    if (j == n_sub - 1) {
                        ptx::umma_commit(&bars->q_empty[qs]);                // the query tile may be replaced
                        if (last_of_head) ptx::umma_commit(&bars->k_empty);  // ... and the key slab
                    }
                }
                __syncwarp();
            }
        }
    } else if (run && warp >= kOwnerWarpG) {
        // ================= owner's reduction =================
        const int owners = owner_count(group_ctas);
        const int my_rows = kTile / owners;                    // rows this CTA owns if rank < owners, at most 32
        const int warp_rows = my_rows > 1 ? my_rows / 2 : 1;   // ... and this warp
        const int n_lanes = 32 / warp_rows;                    // lanes that share a row
        const int sub = lane / warp_rows;                      // this lane takes the pairs of CTAs sub, sub + n_lanes, ...
        const int n_mine = (group_ctas - sub + n_lanes - 1) / n_lanes;  // at least 1 and, since C < 2 owners or C = owners = 128, at most 4
        const int w = warp - kOwnerWarpG;
        const int row = rank * my_rows + w * warp_rows + (lane & (warp_rows - 1));
        const uint4* pairs = xchg + (static_cast<size_t>(group) * group_ctas + sub) * kXchgDepth * kTile + row;
        const bool owner = group_ctas > kMaxDirectCtas && rank < owners && w < my_rows;
        for (int i = 0; owner && i < n_items; ++i) {
            // Entry reuse: row blocks i and i + 8 share entries.
            // Pairs: a warp that posts a pair of block i + 8 has waited for the normalise warps of its CTA to read region
            // (i + 5) mod 3, i.e. for results of block i + 5, whose owners had seen the pairs of every CTA - and this warp reads
            // the pairs of the blocks in order, block i long before.
            // Results: the owner posts a result of block i + 8 after every CTA has posted its pairs of that block, i.e. after
            // the normalise warps of every CTA have read the exponentials of the blocks up to i + 5, with their statistics.
            if (w == 0 && lane == 0) ATTNW_STAMP(22, i);
            const uint32_t tag = tag_base + static_cast<uint32_t>(i) + 1u;
            const uint4* src = pairs + (i & (kXchgDepth - 1)) * kTile;
            uint4 v[4];
            if (!poll_messages<4>(v, n_mine, tag, abort_flag, kSiteGrOwner,
                                  [&](int c) { return src + static_cast<size_t>(c) * n_lanes * kXchgDepth * kTile; }))
                break;
            if (w == 0 && lane == 0) ATTNW_STAMP(23, i);
            float m = fmaxf(fmaxf(__uint_as_float(v[0].x), __uint_as_float(v[1].x)), fmaxf(__uint_as_float(v[2].x), __uint_as_float(v[3].x)));
            for (int off = warp_rows; off < 32; off <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
            float l = 0.0f;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                l += (c < n_mine) ? __uint_as_float(v[c].z) * ptx::ex2_approx(__uint_as_float(v[c].x) - m) : 0.0f;
            for (int off = warp_rows; off < 32; off <<= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
            if (sub == 0) st_message(results + (i & (kXchgDepth - 1)) * kTile + row, m, 1.0f / l, tag);
            if (w == 0 && lane == 0) ATTNW_STAMP(25, i);
        }
    } else if (run && warp < kNormWarp0) {
        // ================= exponential warps: TMEM lane quarter = warp % 4, 32 columns of each slot = warp / 4 =================
        const int part = warp >> 2;
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        // never exactly zero, so that a masked score (-3e38) always lands far below the offset; with scale = 0 every
        // existing score still maps to 2^0
        const float c2 = fmaxf(scale_log2e, 1.0e-30f);
        const uint64_t c2c2 = ptx::pack2(c2, c2);
        float* mbc_all = reinterpret_cast<float*>(smem + L::kMbcOff);
        float2* part_all = reinterpret_cast<float2*>(smem + L::kPartOff);
        uint4* my_msg = xchg + (static_cast<size_t>(blockIdx.x) * kXchgDepth) * kTile + row;
        const bool stamp = warp == 0 && lane == 0;
        (void)stamp;
        bool ok = true;
        for (int i = 0; ok && i < n_items; ++i) {
            const int region = i % kRegions;
            float* mbc = mbc_all + region * kChunksPerBlock * kTile;
            float smax = -3.0e38f, mb = -3.0e38f, l = 0.0f;
            if (stamp) ATTNW_STAMP(0, i);
#pragma unroll 1
            for (int k = 0; k < n_sub; ++k) {
                const int chunk = k * kParts + part;
                const int valid = width - chunk * kChunk;  // columns of this chunk that exist
                const int slot = slot_of(i, k);
                ok = __all_sync(0xffffffffu, fused_wait(&bars->s_full[slot], slot_use(i, k) & 1u, abort_flag, kSiteGrSFull));
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (stamp && k == 0) ATTNW_STAMP(2, i);
                if (stamp) ATTNW_STAMP(17 + 3 * k, i);
                if (valid <= 0) {  // nothing of the chunk is ever stored (the tensor map clips it); the slot's barrier counts every warp
                    if (!kF32) {
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(&bars->s_free[slot]);
                    }
                    continue;
                }
                const uint32_t taddr = t_lane + static_cast<uint32_t>(slot * kSub + part * kChunk);
                uint32_t r[kChunk];
                ptx::tmem_ld_32x32b_x32(taddr, r);
                ptx::tmem_wait_ld();
                if (!kF32) {
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&bars->s_free[slot]);
                }
                if (valid < kChunk) {
#pragma unroll
                    for (int x = 0; x < kChunk; ++x)
                        if (x >= valid) r[x] = 0xff61b1e6u;  // -3.0e38f
                }
                float m0 = __uint_as_float(r[0]), m1 = __uint_as_float(r[1]), m2 = __uint_as_float(r[2]), m3 = __uint_as_float(r[3]);
#pragma unroll
                for (int x = 4; x + 7 < kChunk; x += 8) {
                    m0 = ptx::max3(m0, __uint_as_float(r[x + 0]), __uint_as_float(r[x + 1]));
                    m1 = ptx::max3(m1, __uint_as_float(r[x + 2]), __uint_as_float(r[x + 3]));
                    m2 = ptx::max3(m2, __uint_as_float(r[x + 4]), __uint_as_float(r[x + 5]));
                    m3 = ptx::max3(m3, __uint_as_float(r[x + 6]), __uint_as_float(r[x + 7]));
                }
                m0 = ptx::max3(m0, __uint_as_float(r[kChunk - 4]), __uint_as_float(r[kChunk - 3]));
                m1 = ptx::max3(m1, __uint_as_float(r[kChunk - 2]), __uint_as_float(r[kChunk - 1]));
                const float new_max = ptx::max3(smax, fmaxf(m0, m1), fmaxf(m2, m3));
                const float mb_new = fmaxf(new_max * c2, -3.0e38f);  // finite also while every column so far is masked
                l *= ptx::ex2_approx(mb - mb_new);                   // exactly 1 while the maximum stands
                mb = mb_new;
                smax = new_max;
                if (stamp) ATTNW_STAMP(16 + 3 * k, i);
                uint32_t pk[kChunk / 2];  // bfloat16 output: the exponentials as f16 pairs, in column order
                {
                    const uint64_t off2 = ptx::pack2(-mb, -mb);
                    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
                    // (masked columns hold -3e38 and c2 > 0, so their exponentials are exactly zero)
#pragma unroll
                    for (int x = 0; x < kChunk; x += 2) {
                        float a0, a1;
                        ptx::unpack2(ptx::fma2(ptx::pack2(__uint_as_float(r[x]), __uint_as_float(r[x + 1])), c2c2, off2), a0, a1);
                        a0 = ptx::ex2_approx(a0);
                        a1 = ptx::ex2_approx(a1);
                        if (kF32) {
                            r[x] = __float_as_uint(a0);
                            r[x + 1] = __float_as_uint(a1);
                        } else {
                            pk[x >> 1] = ptx::pack_f16x2(a0, a1);
                        }
                        acc[(x >> 1) & 3] = ptx::add2(acc[(x >> 1) & 3], ptx::pack2(a0, a1));
                    }
                    float s0, s1, s2, s3;
                    ptx::unpack2(ptx::add2(acc[0], acc[1]), s0, s1);
                    ptx::unpack2(ptx::add2(acc[2], acc[3]), s2, s3);
                    l += (s0 + s1) + (s2 + s3);
                }
                if (stamp) ATTNW_STAMP(18 + 3 * k, i);
                if (kF32) {
                    ptx::tmem_st_32x32b_x32(taddr, r);
                } else {
                    // the packed region still holds these columns of row block i - 3 until its normalise warps have read them
                    ok = __all_sync(0xffffffffu, fused_wait(&bars->pk_free[region][chunk >> 1], (static_cast<uint32_t>(i / kRegions) & 1u) ^ 1u, abort_flag, kSiteGrSlotFree));
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
                    ptx::tmem_st_32x32b_x16(t_lane + static_cast<uint32_t>(kPackedCol0 + region * kPackedCols + chunk * (kChunk / 2)), pk);
                }
                if (stamp) ATTNW_STAMP(24 + 2 * k, i);
                mbc[chunk * kTile + row] = mb;  // the offset this chunk's e are relative to
            }
            if (!ok) break;
            part_all[(region * kParts + part) * kTile + row] = make_float2(mb, l);  // this thread's part of the row
            // The last of the four warps to get here merges the parts and posts the row's pair for the group (through L2) at
            // once: the exchange must not wait for a normalise warp to become free.
            __threadfence_block();
            __syncwarp();
            uint32_t before = 0;
            if (lane == 0) before = atomicAdd(&bars->parts_done[region][quarter], 1u);
            before = __shfl_sync(0xffffffffu, before, 0);
            if ((before & (kParts - 1)) == kParts - 1) {
                __threadfence_block();
                const volatile float* pv = reinterpret_cast<const volatile float*>(part_all + region * kParts * kTile + row);
                float pm[kParts], pl[kParts];
#pragma unroll
                for (int x = 0; x < kParts; ++x) {
                    pm[x] = pv[2 * x * kTile];
                    pl[x] = pv[2 * x * kTile + 1];
                }
                const float mc = fmaxf(fmaxf(pm[0], pm[1]), fmaxf(pm[2], pm[3]));
                float lc = 0.0f;
#pragma unroll
                for (int x = 0; x < kParts; ++x) lc += pl[x] * ptx::ex2_approx(pm[x] - mc);
                if (group_ctas > 1)
                    st_message(my_msg + (i & (kXchgDepth - 1)) * kTile, mc, lc, tag_base + static_cast<uint32_t>(i) + 1u);
                else
                    part_all[region * kParts * kTile + row] = make_float2(mc, 1.0f / lc);  // the row's statistics (this thread alone has read the parts)
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars->posted[region]);
            if (stamp) ATTNW_STAMP(4, i);
        }
    } else if (run && warp < kNormWarp0 + 8) {
        // ================= normalise warps: row blocks of parity (warp - 16) / 4, TMEM lane quarter = warp % 4 =================
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t stage = ptx::smem_u32(smem + L::kOutOff + (warp - kNormWarp0) * L::kStages * kStageBytes);
        const uint32_t sw = static_cast<uint32_t>(lane & 7);
        const uint64_t stream_out = ptx::policy_evict_first();
        const float* mbc_all = reinterpret_cast<const float*>(smem + L::kMbcOff) + row;
        const float2* part_all = reinterpret_cast<const float2*>(smem + L::kPartOff) + row;
        const uint4* group_msg = xchg + (static_cast<size_t>(group) * group_ctas * kXchgDepth) * kTile + row;
        uint32_t staged = 0;  // boxes this warp has staged
        const bool stamp = quarter == 0 && lane == 0;
        (void)stamp;
        bool ok = true;
        for (int i = (warp - kNormWarp0) >> 2; ok && i < n_items; i += 2) {
            const int region = i % kRegions;
            const int gi = begin + i, bh = gi / T, row0 = (gi % T) * kTile + quarter * 32;  // first row of this warp
            if (stamp) ATTNW_STAMP(10, i);
            // this CTA's exponentials of the row block are in tensor memory and its chunk offsets in shared memory
            ok = __all_sync(0xffffffffu, fused_wait(&bars->posted[region], static_cast<uint32_t>(i / kRegions) & 1u, abort_flag, kSiteGrPosted));
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (stamp) ATTNW_STAMP(6, i);
            // ---- global statistics of the row ----
            const uint32_t tag = tag_base + static_cast<uint32_t>(i) + 1u;
            const int entry = (i & (kXchgDepth - 1)) * kTile;
            float m_row, inv_l;
            if (group_ctas == 1) {
                const float2 st = part_all[region * kParts * kTile];
                m_row = st.x;
                inv_l = st.y;
            } else if (group_ctas > kMaxDirectCtas) {
                uint4 v[1];
                ok = poll_messages<1>(v, 1, tag, abort_flag, kSiteGrExchange, [&](int) { return results + entry + row; });
                if (!ok) break;
                m_row = __uint_as_float(v[0].x);
                inv_l = __uint_as_float(v[0].z);
            } else {
                // Entry reuse here: a CTA posts block i + 8 after its normalise warps have read the pairs of the blocks up to
                // i + 5, i.e. after EVERY CTA has posted those, which a CTA does after reading the pairs up to block i + 2.
                uint4 v[kMaxDirectCtas];
                ok = poll_messages<kMaxDirectCtas>(v, group_ctas, tag, abort_flag, kSiteGrExchange,
                                                   [&](int c) { return group_msg + static_cast<size_t>(c) * kXchgDepth * kTile + entry; });
                if (!ok) break;
                m_row = __uint_as_float(v[0].x);
#pragma unroll
                for (int c = 1; c < kMaxDirectCtas; ++c) m_row = fmaxf(m_row, __uint_as_float(v[c].x));
                float l_row = 0.0f;
#pragma unroll
                for (int c = 0; c < kMaxDirectCtas; ++c)
                    l_row += (c < group_ctas) ? __uint_as_float(v[c].z) * ptx::ex2_approx(__uint_as_float(v[c].x) - m_row) : 0.0f;
                inv_l = 1.0f / l_row;
            }
            if (stamp) ATTNW_STAMP(11, i);
            // factors of the row's chunks, read before any of the region is handed back (the exponential warps then write the
            // offsets of the next row block there)
            float f[kChunksPerBlock];
#pragma unroll
            for (int c = 0; c < kChunksPerBlock; ++c)
                f[c] = ptx::ex2_approx(mbc_all[(region * kChunksPerBlock + c) * kTile] - m_row) * inv_l;  // (chunks beyond the last key: never stored)
#pragma unroll
            for (int b = 0; b < kMaxBoxes; ++b) {
                if (b < n_boxes) {
                    uint32_t e[kChunk];  // 64 exponentials as f16 pairs, or 32 as float32
                    ptx::tmem_ld_32x32b_x32(t_lane + static_cast<uint32_t>(kF32 ? region * kSlabCols + b * kChunk
                                                                                : kPackedCol0 + region * kPackedCols + b * kChunk), e);
                    ptx::tmem_wait_ld();
                    // the box has been read: the exponentials (float32: the scores) of the next row block may take its place
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (kF32) {
                        const int k = b / (kSub / kBoxCols);
                        if (lane == 0 && (b == n_boxes - 1 || (b + 1) % (kSub / kBoxCols) == 0)) ptx::mbar_arrive(&bars->s_free[region * kSubsPerBlock + k]);
                    } else {
                        if (lane == 0) ptx::mbar_arrive(&bars->pk_free[region][b]);
                    }
                    if (stamp && b == 0) ATTNW_STAMP(12, i);
                    if (stamp && b == 2) ATTNW_STAMP(14, i);
                    // the staging box: the store that used it last must have read it
                    const uint32_t box = stage + (staged % L::kStages) * kStageBytes;
                    ++staged;
                    if (lane == 0) ptx::bulk_wait_group_read<L::kStages - 1>();
                    __syncwarp();
                    if (stamp && b == 2) ATTNW_STAMP(15, i);
                    const uint32_t my_row = box + static_cast<uint32_t>(lane * 128);
#pragma unroll
                    for (int gg = 0; gg < 8; ++gg) {  // one 16-byte piece of the row's 128 bytes
                        uint32_t w[4];
                        if (kF32) {
#pragma unroll
                            for (int x = 0; x < 4; ++x) w[x] = __float_as_uint(__uint_as_float(e[gg * 4 + x]) * f[b]);
                        } else {
                            // p = e * f in float32 from f16 operands (one mixed-precision FMA per element unpacks and
                            // scales); a factor below f16 range rounds to zero, where p < 6e-8 anyway
                            const float fc = f[2 * (b % 4) + (gg >> 2)];
                            const uint32_t fh = ptx::pack_f16x2(fc, fc);
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                float lo, hi;
                                ptx::scale_f16x2(e[gg * 4 + x], fh, lo, hi);
                                w[x] = ptx::pack_bf16x2(lo, hi);
                            }
                        }
                        ptx::st_shared_v4(my_row + ((static_cast<uint32_t>(gg) ^ sw) << 4), w[0], w[1], w[2], w[3]);
                    }
                    if (stamp && b == 2) ATTNW_STAMP(8, i);
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        if (row0 < N) ptx::tma_store_3d(&tm_p, box, col0 + b * kBoxCols, row0, bh, stream_out);
                        ptx::bulk_commit_group();
                    }
                    if (stamp && b == 2) ATTNW_STAMP(9, i);
                }
            }
            if (stamp) ATTNW_STAMP(7, i);
        }
        if (lane == 0) ptx::bulk_wait_group<0>();
    }

    // ---- teardown: every thread of the CTA arrives here, also after a wait gave up ----
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarpG) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

}  // namespace gr
}  // namespace attnw
