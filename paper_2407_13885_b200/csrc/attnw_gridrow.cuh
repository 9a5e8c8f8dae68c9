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
// group.  f16 keeps 11 bits of an exponential, 2.4e-4 relative next to the 2e-3 of the bf16 result, and no more than its
// range: the offset therefore leaves 2^15 of headroom above 1, which keeps those bits down to 2^-29 of the largest of a
// chunk, and the row's factor is applied in float32.  (With the largest at 1 and an f16 factor, weights of 1e-9 .. 1e-6 were
// 0.75 off in relative rms at N = 16384, logits of sigma 16; now 1.7e-3, the rounding of bf16.  It costs 0.5 %: 128 x 4096
// 1090 and 1095 us.)
// Tensor memory, float32 output: two regions of 256 columns; the exponentials replace the scores as float32, and a slot of
// 64 columns goes back to the MMA issuer when its weights have been read.
//
// The CTAs of a group wait for one another, so they must be resident together.  Large hardware clusters do not occupy
// every SM (8 CTAs: 15 clusters of the device's 148 SMs, 16: 7), so large calls are launched cooperatively with one CTA per SM
// and consecutive CTAs form a group; those that clusters serve in as few rounds are launched as clusters, whose launch may
// overlap the kernel in front.  Either way the 16-byte (offset, sum) pair of a row travels through L2 as two 8-byte words that each carry a tag {value, tag, value, tag}; a reader accepts a
// pair once both tags name the row block it is waiting for.  No fence, no flag, no atomics: the tag arrives
// with the value in one 8-byte store.  Every poll is bounded.
//   C = 1          no exchange: the pair stays in shared memory
//   2 <= C <= 4    every CTA reads the C pairs of each row and reduces them redundantly, as the paper's kernel does
//   C > 4          the rows of a block are dealt out to the CTAs; a row's owner reads its C pairs, reduces them once and
//                  posts (M, 1/L) for all (the exchange of Section VIII).  One more hop through L2, but two loads per row
//                  and CTA instead of C, and C may be larger than 16.
//
// Roles of a CTA (896 threads, 28 warps; warp w may touch TMEM lanes 32 (w % 4) ...):
//   warps 0-15   exponentials, four threads per row, thread (row, g) takes columns 32 g ... and 128 + 32 g ...: scores to
//                registers, maximum, offset mb, e = 2^(c s - mb), sum, e back to tensor memory; the thread's (mb, l) to
//                shared memory
//   warps 16-19  normalise the first 128 columns (20-23: the others): a thread owns one row; takes the row's M and 1/L,
//                then per box of 128 bytes a row p = e * 2^(mb - M) / L, rounded to the output type, staged and stored by
//                one TMA store per warp (32 rows x 128 bytes) and box; P is written exactly once
//   warp 24      TMA loads - the CTA's key slab once per head (it stays in shared memory while the group walks the head's row
//                blocks), one query tile per row block - and tcgen05.mma (one elected lane)
//   warps 25-26  merge the four parts of each row and post the row's pair, 64 rows each
//   warp 27      the owner's reduction
//
// What bounds it: nothing alone - at 128 x 4096 x 4096 (d = 128, bfloat16) a block takes 4450 cycles of an SM at a burst, of
// which the special function unit works 2048 and the HBM stream of P would need 2800.  The sixteen exponential warps load,
// reduce and store a slot together, so the unit rests in those phases (1100 of 2150 cycles a slot).  With 8 exponential
// warps of 96 registers, one warp for a row's whole statistics and 16 pairs read by every CTA the same call took 1290 to
// 1340 us in a loop at the power cap, now 1180 to 1240 (1130 -> 1100 at a burst); 12 x 2048 (d = 64) 34.8 -> 30.7,
// 24 x 1000 24.5 -> 18.5.  Instructions count: the waits, votes and address arithmetic around the 3 + 1.6 a score cannot do
// without had been as many again (10.8 a score, then 9.6), and every wait in front of the statistics adds to the time that a
// block's exponentials must be parked, which three regions hide up to some 13000 cycles.
//
// With -DATTNW_TIMELINE=<CTA> one lane per role of that CTA stamps clock64() per row block (events, by index):
//   13 MMA of the block issued | 0 exponentials begin, 2 slot 0 ready, 17/20 load of slot k, 16/19 maximum known,
//   18/21 exponentials of slot k done, 24/26 e stored, 4 parts posted, 1/3 merge begins / pairs posted | 22 owner begins to wait, 23 pairs seen,
//   25 result posted | 10 normalise begins to wait, 6 own CTA done, 11 statistics seen, 12 box 0 read,
//   14/15/8/9 box 1 read / staging free / staged / stored, 7 block done.
#pragma once
#include <cstddef>

#include "attnw_resident.cuh"

namespace attnw {
namespace gr {

constexpr int kSlabCols = 256;                       // key columns per CTA and row block
constexpr int kLandCols = 128;                       // bfloat16: the landing slot = tensor-memory columns [0, 128)
constexpr int kPackedCol0 = kLandCols;               // packed exponentials: columns [128, 512), 128 per region
constexpr int kPackedCols = kSlabCols / 2;           // two f16 per 32-bit column
constexpr int kChunksPerBlock = kSlabCols / kChunk;  // 32-column chunks, each with its own offset
constexpr int kExpWarps = 16;
constexpr int kParts = kExpWarps / 4;                // threads per row
constexpr int kNormWarp0 = kExpWarps;
constexpr int kMmaWarpG = kNormWarp0 + 8;
constexpr int kMergeWarpG = kMmaWarpG + 1;
constexpr int kOwnerWarpG = kMmaWarpG + 3;
constexpr int kThreads = 32 * (kOwnerWarpG + 1);
constexpr int kStageBytes = 32 * 128;                // one staged store box: 32 rows x 128 bytes
constexpr float kHeadroom = 15.0f;                   // bfloat16: exponentials are parked as f16 up to 2^15
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
    uint64_t s_full[8], s_free[8];                          // [slot of tensor memory]: scores ready / slot may be overwritten
    uint64_t pk_free[3];                                    // [region]: the packed exponentials have been read
    uint64_t posted[3];
    uint64_t merged[3];                                     // groups of one CTA: the row statistics are in shared memory
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

// Maximum and sum of the first `n` of four pairs (those beyond repeat one of them).
__device__ __forceinline__ void reduce_pairs(const uint4 (&v)[4], int n, float& m, float& l) {
    m = fmaxf(ptx::max3(__uint_as_float(v[0].x), __uint_as_float(v[1].x), __uint_as_float(v[2].x)), __uint_as_float(v[3].x));
    float t[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) t[c] = c < n ? __uint_as_float(v[c].z) * ptx::ex2_approx(__uint_as_float(v[c].x) - m) : 0.0f;
    l = (t[0] + t[1]) + (t[2] + t[3]);
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
    constexpr int kHalfBoxes = kSlabCols / 2 / kBoxCols;  // store boxes of one normalise warpgroup
    // Columns per MMA slot.  float32: 64, and each half of the exponential warps has slots of its own (32 x 4096 float32 457 ->
    // 439 us against 128); bfloat16: 128 for all of them (64 with a landing slot per half: 128 x 4096 1090 -> 1141 us, since
    // the slots then wait for the one warp that issues twice the instructions).
    constexpr int kSub = kF32 ? 64 : kLandCols;
    constexpr int kSubsPerBlock = kSlabCols / kSub;
    constexpr int kHalves = kF32 ? 2 : 1;
    constexpr int kRegions = kF32 ? 2 : 3;        // row blocks whose exponentials tensor memory holds
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Barriers* bars = reinterpret_cast<Barriers*>(smem + L::kBarOff);
    const uint32_t bar = ptx::smem_u32(bars);
    auto bar_of = [bar](size_t field, int n) { return bar + static_cast<uint32_t>(field) + 8u * static_cast<uint32_t>(n); };
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int group = static_cast<int>(blockIdx.x) / group_ctas;
    const int rank = static_cast<int>(blockIdx.x) % group_ctas;
    if (group >= n_groups) return;  // CTAs beyond the last whole group have no part in the launch
    const int T = (N + kTile - 1) / kTile;                          // row blocks per head
    const int col0 = rank * kSlabCols;                              // first key of this CTA's slab
    const int width = (N - col0 < kSlabCols) ? N - col0 : kSlabCols;  // keys of the slab that exist (>= 1)
    const int n_sub = (width + kSub - 1) / kSub;                    // MMA slots in use, 1..4
    const int n_boxes = (width + kBoxCols - 1) / kBoxCols;          // store boxes in use
    // The group's list: a contiguous range of (head, row block) items, so that the key slab changes rarely.
    const long long begin_ll = static_cast<long long>(total_items) * group / n_groups;
    const long long end_ll = static_cast<long long>(total_items) * (group + 1) / n_groups;
    const int begin = static_cast<int>(begin_ll);
    const int n_items = static_cast<int>(end_ll - begin_ll);
    uint4* const results = xchg + (static_cast<size_t>(n_groups) * group_ctas + group) * kXchgDepth * kTile;

    // ---- set-up ------------------------------------------------------------------------------
    if (threadIdx.x == 0) {
        ptx::grid_dependency_wait();
        const uint32_t prior_failure = *reinterpret_cast<volatile unsigned int*>(&g_attnw_status);  // (arrives meanwhile)
        ptx::mbar_init(&bars->k_full, 1);
        ptx::mbar_init(&bars->k_empty, 1);
        for (int j = 0; j < 8; ++j) {
            ptx::mbar_init(&bars->s_full[j], 1);
            ptx::mbar_init(&bars->s_free[j], kF32 ? 4 : kExpWarps);  // one arrival per warp that reads the slot last
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(&bars->q_full[s], 1);
            ptx::mbar_init(&bars->q_empty[s], 1);
        }
        for (int r = 0; r < 3; ++r) {
            ptx::mbar_init(&bars->pk_free[r], n_boxes > kHalfBoxes ? 8 : 4);  // the normalise warps that have work
            ptx::mbar_init(&bars->posted[r], n_sub >= kHalves ? kExpWarps : kExpWarps / 2);
            ptx::mbar_init(&bars->merged[r], 2);
        }
        bars->abort_flag = 0;
        bars->prior_failure = prior_failure;
        ptx::mbar_fence_init();
    }
    if (warp == kOwnerWarpG && lane == 0) {
        ptx::prefetch_tensormap(&tm_q);
        ptx::prefetch_tensormap(&tm_k);
        ptx::prefetch_tensormap(&tm_p);
    }
    // the parts of rows that no thread writes because their columns do not exist
    for (int x = static_cast<int>(threadIdx.x); x < kRegions * kParts * kTile; x += kThreads)
        if (x / kTile % kParts * kChunk >= width) reinterpret_cast<float2*>(smem + L::kPartOff)[x] = make_float2(-3.0e38f, 0.0f);
    if (warp == kMmaWarpG) {
        ptx::tmem_alloc(&bars->tmem_base, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::grid_dependency_wait();
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    const bool run = bars->prior_failure == 0u && n_items > 0;  // an earlier launch step gave up: skip the work

    // Row blocks use the regions in turn: the region of the list's block i and how often it has been used before, modulo 2.
    struct Turn {
        int region = 0;
        uint32_t parity = 0;
        __device__ __forceinline__ void next(int blocks) {
            region += blocks;
            if (region >= kRegions) {
                region -= kRegions;
                parity ^= 1u;
            }
        }
    };
    // Slot j of a block lands in: bfloat16, the one landing slot; float32, its own columns of the region.
    auto slot_of = [](int region, int j) { return kF32 ? region * kSubsPerBlock + j : 0; };

    if (run && warp == kMmaWarpG) {
        // ================= TMA loads and tcgen05.mma (warp-uniform loop, one elected lane issues) =================
        constexpr uint32_t idesc = ptx::umma_idesc_bf16_f32(kTile, kSub);
        const uint32_t q_addr = ptx::smem_u32(smem + L::kQOff);
        const uint32_t k_addr = ptx::smem_u32(smem + L::kKOff);
        const uint64_t keep = ptx::policy_evict_last();
        const int n_ktiles = (width + kTile - 1) / kTile;
        int bh = begin / T, rb = begin % T;  // of block i
        uint32_t heads = 0;                  // key slabs loaded
        bool ok = true;
        auto load_q = [&](int i, int q_bh, int q_rb) {  // block i's query tile (of the block before last, nothing is left to read)
            if (ptx::elect_one()) {
                ptx::mbar_expect_tx(&bars->q_full[i & 1], static_cast<uint32_t>(L::kTileBytes));
                for (int a = 0; a < L::kAtoms; ++a)
                    ptx::tma_load_3d(smem + L::kQOff + (i & 1) * L::kTileBytes + a * L::kAtomBytes, &tm_q, &bars->q_full[i & 1], a * 64,
                                     q_rb * kTile, q_bh, keep);
            }
            __syncwarp();
        };
        load_q(0, bh, rb);
        Turn turn;
        uint32_t slot_uses = 0;          // bfloat16: of the landing slot
        int issued = 1;                  // query tiles asked for
        for (int i = 0; ok && i < n_items; ++i, turn.next(1)) {
            const int next_bh = rb + 1 == T ? bh + 1 : bh, next_rb = rb + 1 == T ? 0 : rb + 1;
            if (i == 0 || rb == 0) {  // new head: the slab may be replaced once every MMA of the old head has read it
                ok = warp_wait(bar_of(offsetof(Barriers, k_empty), 0), (heads & 1u) ^ 1u, abort_flag, kSiteGrKEmpty);
                if (!ok) break;
                if (ptx::elect_one()) {
                    ptx::mbar_expect_tx(&bars->k_full, static_cast<uint32_t>(n_ktiles * L::kTileBytes));
                    for (int t = 0; t < n_ktiles; ++t)
                        for (int a = 0; a < L::kAtoms; ++a)
                            ptx::tma_load_3d(smem + L::kKOff + a * L::kKAtomBytes + t * L::kAtomBytes, &tm_k, &bars->k_full,
                                             a * 64, col0 + t * kTile, bh, keep);
                }
                __syncwarp();
                ++heads;
                ok = warp_wait(bar_of(offsetof(Barriers, k_full), 0), (heads & 1u) ^ 1u, abort_flag, kSiteGrKFull);
                if (!ok) break;
            }
            ok = warp_wait(bar_of(offsetof(Barriers, q_full), i & 1), static_cast<uint32_t>(i >> 1) & 1u, abort_flag, kSiteGrQFull);
            if (!ok) break;
            for (int j = 0; ok && j < n_sub; ++j) {
                const int slot = slot_of(turn.region, j);
                const uint32_t used = kF32 ? turn.parity : slot_uses++ & 1u;
                ok = warp_wait(bar_of(offsetof(Barriers, s_free), slot), used ^ 1u, abort_flag, kSiteGrSlotFree);
                if (!ok) break;
                ptx::tc_fence_after_sync();
                if (lane == 0 && j == 0) ATTNW_STAMP(13, i);
                const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(slot * kSub);
                // (descriptors: the first of the tile plus a distance in 16-byte units)
                const uint64_t a_desc = ptx::umma_desc_kmajor_sw128(q_addr + static_cast<uint32_t>((i & 1) * L::kTileBytes));
                const uint64_t b_desc = ptx::umma_desc_kmajor_sw128(k_addr + static_cast<uint32_t>(j * kSub * 128));  // keys kSub j ... of every atom
                if (ptx::elect_one()) {
#pragma unroll
                    for (int k = 0; k < D / 16; ++k)
                        ptx::umma_f16_ss(d_tmem, a_desc + static_cast<uint64_t>(((k >> 2) * L::kAtomBytes + (k & 3) * 32) >> 4),
                                         b_desc + static_cast<uint64_t>(((k >> 2) * L::kKAtomBytes + (k & 3) * 32) >> 4), idesc, k > 0 ? 1u : 0u);
                    ptx::umma_commit(&bars->s_full[slot]);
                    if (j == n_sub - 1) {
                        ptx::umma_commit(&bars->q_empty[i & 1]);                               // the query tile may be replaced
                        if (i + 1 == n_items || next_rb == 0) ptx::umma_commit(&bars->k_empty);  // ... and the key slab
                    }
                }
                __syncwarp();
                if (j == 0 && i + 1 < n_items) {  // the next block's query tile, into the place of the previous block's
                    if (i > 0) ok = warp_wait(bar_of(offsetof(Barriers, q_empty), (i + 1) & 1), static_cast<uint32_t>((i - 1) >> 1) & 1u, abort_flag, kSiteGrQEmpty);
                    if (!ok) break;
                    load_q(i + 1, next_bh, next_rb);
                    issued = i + 2;
                }
            }
            bh = next_bh;
            rb = next_rb;
        }
        if (!ok && lane == 0) {
            // Unwinding: let the copies already in flight land before shared memory is released.
            const long long t0 = clock64();
            if (heads > 0)
                while (!ptx::mbar_try_wait(&bars->k_full, (heads - 1u) & 1u) && clock64() - t0 < kWaitLimitCycles / 8) {
                }
            for (int back = 1; back <= 2 && back <= issued; ++back) {
                const int i = issued - back;
                while (!ptx::mbar_try_wait(&bars->q_full[i & 1], static_cast<uint32_t>(i >> 1) & 1u) && clock64() - t0 < kWaitLimitCycles / 4) {
                }
            }
        }
    } else if (run && (warp == kMergeWarpG || warp == kMergeWarpG + 1)) {
        // ================= 64 rows of this CTA's slab: merge the parts, post the pairs =================
        const int row0 = (warp - kMergeWarpG) * 64 + lane;  // and row0 + 32
        uint4* my_msg = xchg + (static_cast<size_t>(blockIdx.x) * kXchgDepth) * kTile + row0;
        float2* part_all = reinterpret_cast<float2*>(smem + L::kPartOff) + row0;
        Turn turn;
        for (int i = 0; i < n_items; ++i, turn.next(1)) {
            if (!warp_wait(bar_of(offsetof(Barriers, posted), turn.region), turn.parity, abort_flag, kSiteGrPosted)) break;
            if (row0 == 0) ATTNW_STAMP(1, i);
            float2* part = part_all + turn.region * kParts * kTile;
            float2 p[2][kParts];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int x = 0; x < kParts; ++x) p[h][x] = part[x * kTile + h * 32];
            float m[2], l[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                m[h] = fmaxf(ptx::max3(p[h][0].x, p[h][1].x, p[h][2].x), p[h][3].x);
                l[h] = (p[h][0].y * ptx::ex2_approx(p[h][0].x - m[h]) + p[h][1].y * ptx::ex2_approx(p[h][1].x - m[h])) +
                       (p[h][2].y * ptx::ex2_approx(p[h][2].x - m[h]) + p[h][3].y * ptx::ex2_approx(p[h][3].x - m[h]));
            }
            if (group_ctas > 1) {
                uint4* msg = my_msg + (i & (kXchgDepth - 1)) * kTile;
                const uint32_t tag = tag_base + static_cast<uint32_t>(i) + 1u;
                st_message(msg, m[0], l[0], tag);
                st_message(msg + 32, m[1], l[1], tag);
            } else {
                part[0] = make_float2(m[0], 1.0f / l[0]);
                part[32] = make_float2(m[1], 1.0f / l[1]);
            }
            if (group_ctas == 1) {
                __syncwarp();
                ptx::mbar_arrive_if(bar_of(offsetof(Barriers, merged), turn.region), lane == 0);
            }
            if (row0 == 0) ATTNW_STAMP(3, i);
        }
    } else if (run && warp == kOwnerWarpG) {
        // ================= the rows of the block that this CTA owns: reduce the group's pairs, post the results =================
        const int owners = owner_count(group_ctas);
        const int my_rows = kTile / owners;                    // at most 32
        const int n_lanes = 32 / my_rows;                      // lanes that share a row
        const int sub = lane / my_rows;                        // this lane takes the pairs of CTAs sub, sub + n_lanes, ...
        const int n_mine = (group_ctas - sub + n_lanes - 1) / n_lanes;  // at least 1 and, since C < 2 owners or C = owners = 128, at most 8
        const int row = rank * my_rows + (lane & (my_rows - 1));
        const uint4* pairs = xchg + (static_cast<size_t>(group) * group_ctas + sub) * kXchgDepth * kTile + row;
        const size_t step = static_cast<size_t>(n_lanes) * kXchgDepth * kTile;
        const bool owner = group_ctas > kMaxDirectCtas && rank < owners;
        for (int i = 0; owner && i < n_items; ++i) {
            // Entry reuse: row blocks i and i + 8 share entries.
            // Pairs: a CTA posts the pairs of block i + 8 after its exponential warps have waited for the normalise warps to read
            // region (i + 5) mod 3, i.e. for results of block i + 5, whose owners had seen the pairs of every CTA - and an
            // owner reads the pairs of the blocks in order, block i long before.
            // Results: the owner posts a result of block i + 8 after every CTA has posted its pairs of that block, i.e. after
            // the normalise warps of every CTA have read the exponentials of the blocks up to i + 5, with their statistics.
            if (lane == 0) ATTNW_STAMP(22, i);
            const uint32_t tag = tag_base + static_cast<uint32_t>(i) + 1u;
            const uint4* src = pairs + (i & (kXchgDepth - 1)) * kTile;
            auto addr = [&](int c) { return src + static_cast<size_t>(c) * step; };
            uint4 v[4];
            if (!poll_messages<4>(v, n_mine, tag, abort_flag, kSiteGrOwner, addr)) break;
            if (lane == 0) ATTNW_STAMP(23, i);
            float m, l;
            reduce_pairs(v, n_mine, m, l);
            if (group_ctas > 4 * n_lanes) {  // (a warp-uniform choice) the other pairs of the lanes
                if (!poll_messages<4>(v, n_mine - 4, tag, abort_flag, kSiteGrOwner, [&](int c) { return addr(c + 4 < n_mine ? c + 4 : n_mine - 1); })) break;
                float m1, l1;
                reduce_pairs(v, n_mine - 4, m1, l1);
                const float mm = n_mine > 4 ? fmaxf(m, m1) : m;
                l = l * ptx::ex2_approx(m - mm) + (n_mine > 4 ? l1 * ptx::ex2_approx(m1 - mm) : 0.0f);
                m = mm;
            }
            // the lanes that share a row are `my_rows` apart
            const float m_lane = m;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1)
                if (off >= my_rows) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
            l *= ptx::ex2_approx(m_lane - m);
#pragma unroll
            for (int off = 1; off < 32; off <<= 1)
                if (off >= my_rows) l += __shfl_xor_sync(0xffffffffu, l, off);
            if (sub == 0) st_message(results + (i & (kXchgDepth - 1)) * kTile + row, m, 1.0f / l, tag);
            if (lane == 0) ATTNW_STAMP(25, i);
        }
    } else if (run && warp < kNormWarp0) {
        // ================= exponential warps: TMEM lane quarter = warp % 4 =================
        const int part = warp >> 2;          // this warp takes columns 128 k + 32 part ..., k = 0, 1
        const int half = kHalves == 2 ? part >> 1 : 0;
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        // never exactly zero, so that a masked score (-3e38) always lands far below the offset; with scale = 0 every
        // existing score still maps to 2^0
        const float c2 = fmaxf(scale_log2e, 1.0e-30f);
        const uint64_t c2c2 = ptx::pack2(c2, c2);
        const uint32_t mbc = ptx::smem_u32(smem + L::kMbcOff) + static_cast<uint32_t>((part * kTile + row) * 4);
        const uint32_t part_addr = ptx::smem_u32(smem + L::kPartOff) + static_cast<uint32_t>((part * kTile + row) * 8);
        const uint32_t lane0 = lane == 0;
        const bool stamp = warp == 0 && lane == 0;
        (void)stamp;
        uint32_t slot_parity = 0;  // bfloat16: of the landing slot's uses
        Turn turn;
        bool ok = half < n_sub;
        for (int i = 0; ok && i < n_items; ++i, turn.next(1)) {
            float smax = -3.0e38f, mb = -3.0e38f, l = 0.0f;
            if (stamp) ATTNW_STAMP(0, i);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (kHalves * k + half >= n_sub) break;
                const int valid = width - (k * 128 + part * kChunk);  // columns of this chunk that exist
                const int slot = slot_of(turn.region, kHalves * k + half);
                ok = warp_wait(bar_of(offsetof(Barriers, s_full), slot), kF32 ? turn.parity : slot_parity, abort_flag, kSiteGrSFull);
                if (!ok) break;
                slot_parity ^= 1u;
                ptx::tc_fence_after_sync();
                if (stamp && k == 0) ATTNW_STAMP(2, i);
                if (stamp) ATTNW_STAMP(17 + 3 * k, i);
                if (valid <= 0) {  // nothing of the chunk is ever stored (the tensor map clips it); the slot's barrier counts every warp
                    if (!kF32) ptx::mbar_arrive_if(bar_of(offsetof(Barriers, s_free), slot), lane0);
                    continue;
                }
                const uint32_t taddr = t_lane + static_cast<uint32_t>(slot * kSub + (kHalves == 2 ? part & 1 : part) * kChunk);
                uint32_t r[kChunk];
                ptx::tmem_ld_32x32b_x32(taddr, r);
                ptx::tmem_wait_ld();
                if (!kF32) {
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    ptx::mbar_arrive_if(bar_of(offsetof(Barriers, s_free), slot), lane0);
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
                smax = ptx::max3(smax, ptx::max3(m0, m1, m2), m3);
                // finite also while every column so far is masked; rounded up, so that no exponential passes 2^kHeadroom
                const float mb_new = fmaxf(kF32 ? smax * c2 : __fmaf_ru(smax, c2, -kHeadroom), -3.0e38f);
                if (k > 0) l *= ptx::ex2_approx(mb - mb_new);     // exactly 1 while the maximum stands
                mb = mb_new;
                if (stamp) ATTNW_STAMP(16 + 3 * k, i);
                uint32_t pk[kChunk / 2];  // bfloat16 output: the exponentials as f16 pairs, in column order
                {
                    const uint64_t off2 = ptx::pack2(-mb, -mb);
                    uint64_t acc[4];
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
                        acc[(x >> 1) & 3] = x < 8 ? ptx::pack2(a0, a1) : ptx::add2(acc[(x >> 1) & 3], ptx::pack2(a0, a1));
                    }
                    float s0, s1;
                    ptx::unpack2(ptx::add2(ptx::add2(acc[0], acc[1]), ptx::add2(acc[2], acc[3])), s0, s1);
                    l += s0 + s1;
                }
                if (stamp) ATTNW_STAMP(18 + 3 * k, i);
                if (kF32) {
                    ptx::tmem_st_32x32b_x32(taddr, r);
                } else {
                    if (k == 0) {  // the packed region still holds row block i - 3 until its normalise warps have read it
                        ok = warp_wait(bar_of(offsetof(Barriers, pk_free), turn.region), turn.parity ^ 1u, abort_flag, kSiteGrSlotFree);
                        if (!ok) break;
                        ptx::tc_fence_after_sync();
                    }
                    ptx::tmem_st_32x32b_x16(t_lane + static_cast<uint32_t>(kPackedCol0 + turn.region * kPackedCols + (k * kParts + part) * (kChunk / 2)), pk);
                }
                if (stamp) ATTNW_STAMP(24 + 2 * k, i);
                ptx::st_shared_f32(mbc + static_cast<uint32_t>((turn.region * kChunksPerBlock + k * kParts) * kTile * 4), mb);  // the offset this chunk's e are relative to
            }
            if (!ok) break;
            // this thread's part of the row (warps without work leave it alone: nothing orders them behind its reader)
            if (part * kChunk < width) ptx::st_shared_v2(part_addr + static_cast<uint32_t>(turn.region * kParts * kTile * 8), mb, l);
            ptx::tmem_wait_st();
            ptx::tc_fence_before_sync();
            __syncwarp();
            ptx::mbar_arrive_if(bar_of(offsetof(Barriers, posted), turn.region), lane0);
            if (stamp) ATTNW_STAMP(4, i);
        }
    } else if (run && warp < kNormWarp0 + 8) {
        // ================= normalise warps: keys of slot (warp - 16) / 4, TMEM lane quarter = warp % 4 =================
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t t_lane = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t stage = ptx::smem_u32(smem + L::kOutOff + (warp - kNormWarp0) * L::kStages * kStageBytes);
        const uint32_t sw = static_cast<uint32_t>(lane & 7);
        const uint64_t stream_out = ptx::policy_evict_first();
        const float* mbc_all = reinterpret_cast<const float*>(smem + L::kMbcOff) + row;
        const float2* part_all = reinterpret_cast<const float2*>(smem + L::kPartOff) + row;
        const uint4* group_msg = xchg + (static_cast<size_t>(group) * group_ctas * kXchgDepth) * kTile + row;
        uint32_t box = stage;  // the staging box to be used next
        const uint32_t lane0 = lane == 0;
        const bool stamp = warp == kNormWarp0 && lane == 0;
        (void)stamp;
        const int box0 = ((warp - kNormWarp0) >> 2) * kHalfBoxes;  // the first box of this warpgroup
        int bh = begin / T, rb = begin % T;
        Turn turn;
        bool ok = box0 < n_boxes;
        for (int i = 0; ok && i < n_items; ++i, turn.next(1)) {
            const int region = turn.region;
            if (stamp) ATTNW_STAMP(10, i);
            // this CTA's exponentials of the row block are in tensor memory and its chunk offsets in shared memory
            ok = warp_wait(bar_of(offsetof(Barriers, posted), region), turn.parity, abort_flag, kSiteGrPosted);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            if (stamp) ATTNW_STAMP(6, i);
            // ---- global statistics of the row ----
            const uint32_t tag = tag_base + static_cast<uint32_t>(i) + 1u;
            const int entry = (i & (kXchgDepth - 1)) * kTile;
            float m_row, inv_l;
            if (group_ctas == 1) {
                ok = warp_wait(bar_of(offsetof(Barriers, merged), region), turn.parity, abort_flag, kSiteGrPosted);
                if (!ok) break;
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
            const int row0 = rb * kTile + quarter * 32;  // first row of this warp
            // factors of the row's chunks, read before any of the region is handed back (the exponential warps then write the
            // offsets of the next row block there)
            float f[kParts];
#pragma unroll
            for (int c = 0; c < kParts; ++c)
                f[c] = ptx::ex2_approx(mbc_all[(region * kChunksPerBlock + box0 * kBoxCols / kChunk + c) * kTile] - m_row) * inv_l;  // (chunks beyond the last key: never stored)
#pragma unroll
            for (int b = 0; b < kHalfBoxes; ++b) {
                if (box0 + b < n_boxes) {
                    uint32_t e[kChunk];  // 64 exponentials as f16 pairs, or 32 as float32
                    ptx::tmem_ld_32x32b_x32(t_lane + static_cast<uint32_t>((kF32 ? region * kSlabCols : kPackedCol0 + region * kPackedCols) +
                                                                           (box0 + b) * kChunk), e);
                    ptx::tmem_wait_ld();
                    // the last of a slot (float32) or of this warpgroup's boxes has been read: the next row block may take their place
                    const bool last = b == kHalfBoxes - 1 || box0 + b == n_boxes - 1;
                    if (last || (kF32 && (b + 1) % (kSub / kBoxCols) == 0)) {
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        ptx::mbar_arrive_if(kF32 ? bar_of(offsetof(Barriers, s_free), region * kSubsPerBlock + (box0 + b) / (kSub / kBoxCols))
                                                 : bar_of(offsetof(Barriers, pk_free), region), lane0);
                    }
                    if (stamp && b == 0) ATTNW_STAMP(12, i);
                    if (stamp && b == 1) ATTNW_STAMP(14, i);
                    // the staging box: the store that used it last must have read it (lane 0 has issued them all)
                    ptx::bulk_wait_group_read<L::kStages - 1>();
                    __syncwarp();
                    if (stamp && b == 1) ATTNW_STAMP(15, i);
                    const uint32_t my_row = box + static_cast<uint32_t>(lane * 128);
#pragma unroll
                    for (int gg = 0; gg < 8; ++gg) {  // one 16-byte piece of the row's 128 bytes
                        uint32_t w[4];
                        if (kF32) {
#pragma unroll
                            for (int x = 0; x < 4; ++x) w[x] = __float_as_uint(__uint_as_float(e[gg * 4 + x]) * f[b]);
                        } else {
                            const float fc = f[(2 * b + (gg >> 2)) % kParts];
                            const uint64_t ff = ptx::pack2(fc, fc);
#pragma unroll
                            for (int x = 0; x < 4; ++x) {
                                float lo, hi;
                                ptx::unpack_f16x2(e[gg * 4 + x], lo, hi);
                                ptx::unpack2(ptx::mul2(ptx::pack2(lo, hi), ff), lo, hi);
                                w[x] = ptx::pack_bf16x2(lo, hi);
                            }
                        }
                        ptx::st_shared_v4(my_row + ((static_cast<uint32_t>(gg) ^ sw) << 4), w[0], w[1], w[2], w[3]);
                    }
                    if (stamp && b == 1) ATTNW_STAMP(8, i);
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    ptx::tma_store_3d_if(lane0 & static_cast<uint32_t>(row0 < N), &tm_p, box, col0 + (box0 + b) * kBoxCols, row0, bh, stream_out);
                    ptx::bulk_commit_group();
                    box = box == stage + (L::kStages - 1) * kStageBytes ? stage : box + kStageBytes;
                    if (stamp && b == 1) ATTNW_STAMP(9, i);
                }
            }
            if (++rb == T) {
                rb = 0;
                ++bh;
            }
            if (stamp) ATTNW_STAMP(7, i);
        }
        ptx::bulk_wait_group<0>();
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
