// Fused attention O = Softmax(scale * Q K^T) V for sm_100a in ONE pass over the keys: Attention(Q, K, V) of
// Section IV (the product with V is the paper's future work, Section VIII) with the online form of Eq. 1.
//
// A CTA holds two units that share its tensor pipe and its special function units: two query tiles of 128 rows over all
// key tiles, or (split) ONE query tile, unit 0 over the even and unit 1 over the odd key tiles, merged at the end; or the
// 2 G units of a cluster of G CTAs share one query tile, unit u over the key tiles u, u + 2 G, ...
// Per step j and unit q:
//   MMA 1     S = Q K_j^T                         128 x 128 fp32 in tensor memory
//   Softmax   two threads per row, 64 columns each: a thread takes its scores to registers (the buffer is handed back
//             at once, so the next MMA 1 runs meanwhile); the two tell each other their maximum through shared memory; the units
//             take turns at the exponentials;
//             p = 2^(c s - mb) with the row's offset mb; l += sum p; P (bf16) becomes the A operand of MMA 2 in tensor memory
//   MMA 2     O_q += P V_j                        128 x d fp32 in tensor memory; V_j as TMA delivers it
//             ([128 keys x d], an MN-major B operand)
// The offset mb of a row follows its running maximum lazily: it moves only when the maximum has grown by more than 8
// (in the base-2 exponent), and then O's row and l are multiplied by 2^(mb_old - mb_new) - after the first tiles
// this is rare, and weights stay below 2^8.  The division by l happens once, in the epilogue.  One exponential and
// two MMA passes per element.  (An offset that follows one step late, so that no exponential waits for a maximum, took 1.18 ms
// instead of 1.01 at 128 x 4096, d = 128: 88 bytes of spills, and the maximum is not what the unit waits for.)
// What bounds it: in a loop of large calls, the power cap; at a burst, the chain of the Softmax warps' step (d = 128: 3100 cycles
// of which the special function units and the tensor pipe need 2048 each).  Operand fetch from shared memory holds up
// the tensor pipe, and the issuers' waits keep it idle (two_issuers), so:
//   * P goes through tensor memory (through shared memory its port was busy 3072 of 4200 cycles a step): 128 x 4096, d = 64
//     839 -> 801 us; d = 128 985 -> 941 at a burst, 1106 -> 1056 in a loop.  d = 64 has room for the scores of both units beside P
//     and O.  d = 128 has one buffer of scores: the units are half a step apart and hold it only from MMA 1 until their
//     scores are in registers, less than half a step.
//   * The two threads of a row exchange maxima (each read the other's scores too, which held the buffer longer), and the
//     room of P's tiles makes the ring of K and V a stage longer: d = 128 941 -> 910 and 1057 -> 1027; d = 64 793 -> 768;
//     12 x 1021, d = 64 13.0 -> 12.1.
//   * The units take turns at the exponentials (turns), and units of one query tile have an issuing warp for the scores and one for the products
//     (two_issuers): 12 x 1021, d = 64 11.9 -> 11.2, 3 x 12766 257 -> 236, 13 x 7115, d = 128 336 -> 318; 36 drawn sizes 1.035 times as fast.
// Slower: the issuer asking for both barriers of a set of MMAs at once, and one election for MMAs and release (d = 128 977 -> 996 us, an
// issuer that finds the second one not ready asks for the first again); the wait for the previous product put off until half of the weights are there (d = 64 780 -> 821 us, d = 128 no change);
// one thread per row, 8 Softmax warps of 168 registers (d = 64 795 -> 1000: a lone warp of a scheduler gets half of
// its special function unit); products before scores (780 -> 978); 1/8 or 1/4 of the exponentials by a polynomial of degree 5 on
// the FMA pipes (d = 64 778 -> 776, 790; d = 128 965 -> 984, 1002 in a loop); CTAs that stay for several row blocks and store
// O from registers (d = 128 905 -> 896 at a burst, d = 64 800 -> 843).
// Valid for any N >= 1, d in {64, 128}; Q, K, V, O bf16 [B, H, N, d].
#pragma once
#include <cstddef>

#include "attn_fused.cuh"

namespace attnw {
namespace av1 {

constexpr int kSmWarps = 16;      // Softmax warps: unit (2) x column half (2) x TMEM lane quarter (4)
constexpr int kProducer = 16;
constexpr int kMma = 17;
constexpr int kMmaProduct = 18;   // two_issuers: the products' issuer
constexpr int kMaxCluster = 4;    // CTAs that share a query tile (of 8, 15 clusters fit, and a call that needs them has 16 tiles)
constexpr int kPassAt = 4;        // of the 8 groups of 8 exponentials: behind which the other unit's turn begins
constexpr float kLazy = 8.0f;     // the offset follows the maximum only when it has grown by more than this

enum : uint32_t {  // wait sites of this kernel (low byte of the status word)
    kSiteProducerEmpty = 96,
    kSiteMmaQ = 97,
    kSiteMmaKFull = 98,
    kSiteMmaSFree = 99,
    kSiteMmaPFull = 100,
    kSiteSFull = 101,
    kSitePFree = 102,
    kSiteOFull = 103,
    kSiteOutFilled = 104,
    kSiteLFull = 105,
    kSiteMaxFull = 106,
    kSitePairsIn = 107,
};

constexpr int kUnitStats = 4 * kTile;

// How the keys of a query tile are worked on.
enum Mode { kWhole, kSplit, kCluster };

template <int D>
struct Smem {
    static constexpr int kAtoms = D / 64;
    static constexpr int kAtomBytes = kTile * 128;             // 128 rows x 128 bytes
    static constexpr int kTileBytes = kAtoms * kAtomBytes;     // a Q, K or V tile
    static constexpr int kStages = (D == 128) ? 4 : 6;         // ring of K / V tiles (128 keys x d)
    // Tensor memory: d = 64 has room for scores, O and P (the product's A operand) of both units; d = 128 for P and O of
    // both and ONE buffer of scores, which the units use in turn.
    static constexpr bool kSharedS = D == 128;
    // A second warp issues the products: an issuer spends 200 to 550 cycles on the waits in front of each set of MMAs, 1360 of a
    // step's 3450 at d = 128, and nothing of the other kind was queued meanwhile.  128 x 4096 902 -> 856 us at a burst, 1012 -> 950
    // in a loop; 12 x 2048 34.8 -> 32.4.  At d = 64 the MMAs take half as long: with two query tiles the exponentials set the pace
    // (780 us with one issuer, 811 with two), but units of one query tile have K and V tiles of their own and twice the waits (12 x 1021 12.2 ->
    // 11.2, 4 x 13233 302 -> 261).
    static __host__ __device__ constexpr bool two_issuers(Mode m) { return D == 128 || m != kWhole; }
    // The two units take turns at the exponentials.  The warps of a lane quarter, two of each unit, share a scheduler and its special function
    // unit, and left alone they fall into step: all in their exponentials (twice as long), then all in their waits and maxima.  The turn
    // passes when 5 of 8 groups of exponentials are issued: what is left of them covers the hand-over.  us per call without turns -> with
    // them (behind 4, 6 or all groups): d = 64, 128 x 4096 756 -> 746 (785, 810, 872), 4 x 13233 274 -> 261; d = 128, 9 x 6108 175 -> 167, 3 x 13719
    // 334 -> 314, 2 x 363 8.1 -> 7.6; not for two query tiles at d = 128, whose scores alternate anyway (956 -> 963).
    static __host__ __device__ constexpr bool turns(Mode m) { return D == 64 || m != kWhole; }
    static __host__ __device__ constexpr int threads(Mode m) { return two_issuers(m) ? 608 : 576; }
    static __host__ __device__ constexpr uint32_t s_col(int q) { return kSharedS ? 0u : static_cast<uint32_t>(q * 256); }
    static __host__ __device__ constexpr uint32_t p_col(int q) { return kSharedS ? 128u + static_cast<uint32_t>(q * 64) : static_cast<uint32_t>(q * 256 + 192); }
    static __host__ __device__ constexpr uint32_t o_col(int q) { return kSharedS ? 256u + static_cast<uint32_t>(q * 128) : static_cast<uint32_t>(q * 256 + 128); }
    static constexpr int kQOff = 0;                            // two query tiles; split: one, and one more stage of the ring
    static constexpr int kKOff = kQOff + 2 * kTileBytes;
    static constexpr int kStatOff = kKOff + kStages * kTileBytes;  // per unit: maxima, float [2 steps][2 halves][128 rows]; at the end sums and offset
    static constexpr int kPairOff = kStatOff + 2 * kUnitStats * 4;  // clusters: float2 [CTA][128 rows], (offset, sum) of each CTA's part
    static constexpr int kBarOff = kPairOff + kMaxCluster * kTile * 8;
    static constexpr int kBytes = kBarOff + 512;
    static constexpr int kDynamicBytes = kBytes + 1024;
};
static_assert(Smem<128>::kDynamicBytes <= 227 * 1024, "shared memory budget");

struct Barriers {
    uint64_t q_full;
    uint64_t k_full[7], k_empty[7];
    uint64_t s_full[2], s_free[2];  // per unit: scores written / read into registers (8 warps)
    uint64_t p_full[2], p_free[2];  // per unit: P written (8 warps) / read by its MMAs
    uint64_t o_full[2];             // per unit: every product complete
    uint64_t max_full[2][4];        // per unit and lane quarter, without turns: the maxima of both halves are in shared memory (2 warps)
    uint64_t l_full[2];             // per query tile: the row statistics of its warps are in shared memory
    uint64_t out_filled[2];
    uint64_t pairs_in;              // clusters: the pairs of every CTA have arrived
    uint32_t tmem_base;
    uint32_t abort_flag;
};
static_assert(sizeof(Barriers) <= 512, "barrier block must fit its slot");

// The bounded wait of the other kernels, but expanded in place: where a thread holds a row of scores in registers,
// a call would spill them around it.
__device__ __forceinline__ bool wait_in_place(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (uint32_t spin = 1;; ++spin) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if ((spin & 63u) == 0) {
            if (*abort_flag) return false;
            if (clock64() - t0 > kWaitLimitCycles) {
                *abort_flag = 1;
                atomicCAS(&g_attnw_status, 0u, 0x80000000u | site);
                return false;
            }
        }
    }
}

template <int D, Mode M>
__global__ void __launch_bounds__(Smem<D>::threads(M), 1)
attn_onepass_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o, int N,
                    int row_blocks_per_head, float scale_log2e, __nv_bfloat16* O, int cluster_ctas, int first_block) {
    using L = Smem<D>;
    constexpr bool split = M != kWhole;
    constexpr bool two_issuers = L::two_issuers(M);
    constexpr bool turns = L::turns(M);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Barriers* bars = reinterpret_cast<Barriers*>(smem + L::kBarOff);
    const uint32_t bar = ptx::smem_u32(bars);
    auto bar_of = [bar](size_t field, int n) { return bar + static_cast<uint32_t>(field) + 8u * static_cast<uint32_t>(n); };
    volatile uint32_t* abort_flag = &bars->abort_flag;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int G = M == kCluster ? cluster_ctas : 1;  // CTAs that share a query tile
    const int rank = M == kCluster ? static_cast<int>(ptx::cluster_ctarank()) : 0;
    const int block = first_block + static_cast<int>(blockIdx.x) / G;  // of those of all heads
    const int bh = block / row_blocks_per_head;
    const int row0 = (block % row_blocks_per_head) * (split ? kTile : kRowsPerCta);
    const int T = (N + kTile - 1) / kTile;  // key tiles
    // The key tiles of a unit: all of them, or one in 2 G.
    const int units = split ? 2 * G : 1;
    auto key_tile = [&](int j, int q) { return split ? units * j + 2 * rank + q : j; };
    const int steps[2] = {split ? (T - 2 * rank + units - 1) / units : T,
                          split ? (T - 2 * rank + units - 2) / units : (row0 + kTile < N ? T : 0)};
    constexpr int kStages = L::kStages + (split ? 1 : 0);
    auto stage_offset = [](int s) { return !split || s < L::kStages ? L::kKOff + s * L::kTileBytes : L::kQOff + L::kTileBytes; };

    // ---- set-up ------------------------------------------------------------------------------
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bars->q_full, 1);
        for (int s = 0; s < 7; ++s) {
            ptx::mbar_init(&bars->k_full[s], 1);
            ptx::mbar_init(&bars->k_empty[s], 1);
        }
        for (int q = 0; q < 2; ++q) {
            ptx::mbar_init(&bars->s_full[q], 1);
            ptx::mbar_init(&bars->s_free[q], 8);
            ptx::mbar_init(&bars->p_full[q], 8);
            ptx::mbar_init(&bars->p_free[q], 1);
            ptx::mbar_init(&bars->o_full[q], 1);
            for (int w = 0; w < 4; ++w) ptx::mbar_init(&bars->max_full[q][w], 2);
            ptx::mbar_init(&bars->l_full[q], split ? 16 : 8);
            ptx::mbar_init(&bars->out_filled[q], split ? 15 : 7);
        }
        if constexpr (M == kCluster) {
            ptx::mbar_init(&bars->pairs_in, 1);
            ptx::mbar_expect_tx(&bars->pairs_in, static_cast<uint32_t>(G * kTile * 8));
        }
        bars->abort_flag = 0;
        ptx::mbar_fence_init();
    }
    if (warp == kProducer && lane == 0) {
        ptx::prefetch_tensormap(&tm_q);
        ptx::prefetch_tensormap(&tm_k);
        ptx::prefetch_tensormap(&tm_v);
        ptx::prefetch_tensormap(&tm_o);
    }
    if (warp == kMma) {
        ptx::tmem_alloc(&bars->tmem_base, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::grid_dependency_wait();
    ptx::tc_fence_before_sync();
    __syncthreads();
    if constexpr (M == kCluster) {  // every CTA runs, with its barriers in place, before anyone writes into a peer
        ptx::cluster_arrive_relaxed();
        ptx::cluster_wait_acquire();
    }
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = bars->tmem_base;
    int loads = 0;  // producer: ring entries asked for

    if (warp == kProducer) {
        // ================= TMA producer: Q once, then the K and V tiles in the order the MMA issuer reads them =========
        // Two query tiles at d = 128: the whole warp walks the list and an elected lane issues (a lone lane takes 300 cycles a tile: 2 x 97
        // 6.4 -> 6.2 us).  Otherwise a lone lane (3 x 863, d = 64 10.06 us, the whole warp 10.16; 3 x 802, d = 128 11.05 and 11.15).
        constexpr bool whole_warp = D == 128 && M == kWhole;
        if (whole_warp || lane == 0) {
            const uint64_t keep = ptx::policy_evict_last();
            auto issues = [&]() { return !whole_warp || ptx::elect_one(); };
            const int q_tiles = (!split && steps[1] > 0) ? 2 : 1;
            if (issues()) {
                ptx::mbar_expect_tx(&bars->q_full, static_cast<uint32_t>(q_tiles * L::kTileBytes));
                for (int q = 0; q < q_tiles; ++q)
                    for (int a = 0; a < L::kAtoms; ++a)
                        ptx::tma_load_3d(smem + L::kQOff + q * L::kTileBytes + a * L::kAtomBytes, &tm_q, &bars->q_full, a * 64,
                                         row0 + q * kTile, bh, keep);
            }
            if (whole_warp) __syncwarp();
            int n = 0;
            bool ok = true;
            auto load = [&](const CUtensorMap* map, int kt) {
                if (!ok) return;
                const int s = n % kStages;
                const uint32_t parity = (static_cast<uint32_t>(n / kStages) & 1u) ^ 1u;
                ok = whole_warp ? warp_wait(bar_of(offsetof(Barriers, k_empty), s), parity, abort_flag, kSiteProducerEmpty)
                                : fused_wait(&bars->k_empty[s], parity, abort_flag, kSiteProducerEmpty);
                if (!ok) return;
                if (issues()) {
                    ptx::mbar_expect_tx(&bars->k_full[s], static_cast<uint32_t>(L::kTileBytes));
                    for (int a = 0; a < L::kAtoms; ++a)
                        ptx::tma_load_3d(smem + stage_offset(s) + a * L::kAtomBytes, map, &bars->k_full[s], a * 64, kt * kTile, bh, keep);
                }
                if (whole_warp) __syncwarp();
                ++n;
            };
            const int lists = split ? 2 : 1;  // units that have key tiles of their own
            for (int j = -1; ok && j < steps[0]; ++j) {
                for (int q = 0; q < lists; ++q) {
                    if (j + 1 < steps[q]) load(&tm_k, key_tile(j + 1, q));
                    if (j >= 0 && j < steps[q]) load(&tm_v, key_tile(j, q));
                }
            }
            loads = n;
        }
        __syncwarp();
    } else if (warp == kMma || (two_issuers && warp == kMmaProduct)) {
        // ================= MMA issuers (warp-uniform loops, one elected lane issues): of scores, of products, or of both =================
        constexpr uint32_t idesc_s = ptx::umma_idesc_bf16_f32(kTile, kTile);
        constexpr uint32_t idesc_o = ptx::umma_idesc_bf16_f32(kTile, D) | (1u << 16);  // B operand MN-major
        const uint32_t base = ptx::smem_u32(smem);
        // Did an earlier launch give up?  Then this one computes and writes nothing: looked at in front of the first MMA, when it has
        // arrived beside the first loads (in front of the set-up's barrier: 3 x 128 5.04 us, now 4.91; 7 x 64, d = 128 6.10, 5.93; 12 x 1021 11.2, 11.1).
        const uint32_t prior_failure = *reinterpret_cast<volatile unsigned int*>(&g_attnw_status);
        bool ok = warp_wait(bar_of(offsetof(Barriers, q_full), 0), 0, abort_flag, kSiteMmaQ);
        if (__any_sync(0xffffffffu, prior_failure != 0u)) {
            *abort_flag = 1;
            ok = false;
            if constexpr (M == kCluster) tell_peers(&bars->abort_flag, G);
        }
        int n = 0;            // next ring entry, in step with the producer
        auto arrived = [&]() {
            ok = ok && warp_wait(bar_of(offsetof(Barriers, k_full), n % kStages), static_cast<uint32_t>(n / kStages) & 1u, abort_flag, kSiteMmaKFull);
        };
        auto release = [&]() {  // the entry may be replaced once the MMAs issued so far are complete
            if (ptx::elect_one()) ptx::umma_commit(&bars->k_empty[n % kStages]);
            __syncwarp();
            ++n;
        };
        int last_q = 0, last_j = -1;  // kSharedS: whose scores the buffer holds
        auto scores = [&](int q, int j) {  // S of step j
            // the row threads have the scores that are in the buffer in registers
            const int before_q = L::kSharedS ? last_q : q, before_j = L::kSharedS ? last_j : j - 1;
            ok = ok && warp_wait(bar_of(offsetof(Barriers, s_free), before_q), static_cast<uint32_t>(before_j) & 1u, abort_flag, kSiteMmaSFree);
            if (!ok) return;
            last_q = q;
            last_j = j;
            ptx::tc_fence_after_sync();
            const uint32_t d_tmem = tmem_base + L::s_col(q);
            // (descriptors: the first of the tile plus a distance in 16-byte units)
            const uint64_t a_desc = ptx::umma_desc_kmajor_sw128(base + L::kQOff + (split ? 0u : static_cast<uint32_t>(q * L::kTileBytes)));
            const uint64_t b_desc = ptx::umma_desc_kmajor_sw128(base + static_cast<uint32_t>(stage_offset(n % kStages)));
            if (ptx::elect_one()) {
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
                    const uint64_t off = static_cast<uint64_t>(((k >> 2) * L::kAtomBytes + (k & 3) * 32) >> 4);
                    ptx::umma_f16_ss(d_tmem, a_desc + off, b_desc + off, idesc_s, k > 0 ? 1u : 0u);
                }
                ptx::umma_commit(&bars->s_full[q]);
            }
            __syncwarp();
        };
        auto product = [&](int q, int j) {  // O += P V of step j
            ok = ok && warp_wait(bar_of(offsetof(Barriers, p_full), q), static_cast<uint32_t>(j) & 1u, abort_flag, kSiteMmaPFull);
            if (!ok) return;
            ptx::tc_fence_after_sync();
            const uint32_t o_tmem = tmem_base + L::o_col(q), p_tmem = tmem_base + L::p_col(q);
            const uint64_t b_desc = av::umma_desc_mnmajor_sw128(base + static_cast<uint32_t>(stage_offset(n % kStages)), L::kAtomBytes);
            if (ptx::elect_one()) {
#pragma unroll
                for (int kk = 0; kk < kTile / 16; ++kk)  // 16 keys per instruction
                    ptx::umma_f16_ts(o_tmem, p_tmem + static_cast<uint32_t>(kk * 8), b_desc + static_cast<uint64_t>(kk * 16 * 128 >> 4), idesc_o,
                                     (j > 0 || kk > 0) ? 1u : 0u);
                ptx::umma_commit(&bars->p_free[q]);
                if (j + 1 == steps[q]) ptx::umma_commit(&bars->o_full[q]);
            }
            __syncwarp();
        };
        // The scores of step j + 1 first: the tensor pipe computes them while the row threads exponentiate step j.  The two
        // units alternate (with two issuers, because the scores take turns at their buffer) - scores of one, product of one, scores of
        // the other, product of the other - which keeps their row threads half a step apart (d = 64, 128 x 4096: 888 -> 841 us against
        // both scores first).
        if constexpr (two_issuers) {
            const bool for_scores = warp == kMma;
            for (int j = -1; ok && j < steps[0]; ++j) {
                for (int q = 0; ok && q < (split ? 2 : 1); ++q) {
                    if (j + 1 < steps[q]) {  // K of step j + 1
                        if (for_scores) {
                            arrived();
                            scores(q, j + 1);
                            if (!split && steps[1] > 0) scores(1, j + 1);
                            release();
                        } else {
                            ++n;
                        }
                    }
                    if (j >= 0 && j < steps[q]) {  // V of step j
                        if (!for_scores) {
                            arrived();
                            product(q, j);
                            if (!split && steps[1] > 0) product(1, j);
                            release();
                        } else {
                            ++n;
                        }
                    }
                }
            }
        } else {
            static_assert(two_issuers || !split, "one issuer: two query tiles");
            for (int j = -1; ok && j < steps[0]; ++j) {
                const bool next = j + 1 < T;
                const int k_entry = n, v_entry = next ? n + 1 : n;  // K of step j + 1, V of step j
                if (next) {
                    arrived();
                    scores(0, j + 1);
                }
                n = v_entry;
                if (ok && j >= 0) {
                    arrived();
                    product(0, j);
                }
                if (ok && next) {
                    n = k_entry;
                    if (steps[1] > 0) scores(1, j + 1);
                    release();
                }
                if (ok && j >= 0) {
                    n = v_entry;
                    if (steps[1] > 0) product(1, j);
                    release();
                }
            }
        }
    } else if (warp < kSmWarps) {
        // ================= Softmax warps: two threads per query row, 64 key columns of a tile each =================
        const int q = warp >> 3;
        const int half = (warp >> 2) & 1;
        const int quarter = warp & 3;
        const uint32_t t_quarter = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t t_own = t_quarter + L::s_col(q) + static_cast<uint32_t>(half * kHalf);
        const uint32_t o_own = t_quarter + L::o_col(q) + static_cast<uint32_t>(half * (D / 2));  // this thread's D/2 columns of O
        const float c2 = scale_log2e;
        const uint64_t c2c2 = ptx::pack2(c2, c2);
        const int row = quarter * 32 + lane;
        // The two threads of a row tell each other their maximum through shared memory, even and odd steps in places of their own
        // (a thread is at most one step ahead of the other).
        float* const stats = reinterpret_cast<float*>(smem + L::kStatOff) + q * kUnitStats;
        const uint32_t max_own = ptx::smem_u32(stats + half * kTile + row), max_other = ptx::smem_u32(stats + (half ^ 1) * kTile + row);
        const uint32_t lane0 = lane == 0;
        const uint32_t sw = static_cast<uint32_t>(lane & 7);
        const uint32_t p_own = t_quarter + L::p_col(q) + static_cast<uint32_t>(half * 32);  // its 64 keys of P
        float smax = -3.0e38f;  // running maximum of the raw scores of this row (all columns)
        float mb = -3.0e38f;    // the offset the weights, l and O's row are relative to (follows smax * c2 lazily)
        float l = 0.0f;         // sum of this thread's weights
        bool ok = true;

        const int my_steps = q == 0 ? steps[0] : steps[1], other_steps = q == 0 ? steps[1] : steps[0];
        // turns: unit 0's step 0, unit 1's step 0, unit 0's step 1, ... of those that both units have; the barrier of a turn is the one that the
        // two threads of a row exchange their maxima by.  Every warp takes part in all of them, also after a wait has given up.
        const uint32_t turn_own = static_cast<uint32_t>(1 + q * 4 + quarter), turn_other = static_cast<uint32_t>(1 + (q ^ 1) * 4 + quarter);
        const int behind = q == 0 ? 1 : 0;  // a step waits for the other unit's step so many before
        auto take_turn = [&](int j) {
            if (turns) ptx::named_sync(turn_own, j >= behind && j - behind < other_steps ? 128u : 64u);
        };
        auto pass_turn = [&](int j) {
            if (turns && j + 1 - behind < other_steps) ptx::named_arrive(turn_other, 128u);
        };
        for (int j = 0; j < my_steps; ++j) {
            if (ok) ok = warp_wait(bar_of(offsetof(Barriers, s_full), q), static_cast<uint32_t>(j) & 1u, abort_flag, kSiteSFull);
            if (!ok) {
                take_turn(j);
                pass_turn(j);
                continue;
            }
            ptx::tc_fence_after_sync();
            const int valid = N - key_tile(j, q) * kTile;  // key columns of this tile that exist
            // ---- this thread's 64 scores into registers; the buffer goes back to the MMA issuer at once ----
            float s[kHalf];
            {
                uint32_t r0[kChunk], r1[kChunk];
                ptx::tmem_ld_32x32b_x32(t_own, r0);
                ptx::tmem_ld_32x32b_x32(t_own + kChunk, r1);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < kChunk; ++i) {
                    s[i] = __uint_as_float(r0[i]);
                    s[kChunk + i] = __uint_as_float(r1[i]);
                }
            }
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars->s_free[q]);
            if (valid < kTile) {
#pragma unroll
                for (int i = 0; i < kHalf; ++i)
                    if (half * kHalf + i >= valid) s[i] = -3.0e38f;
            }
            // ---- row maximum, lazy offset ----
            float m0 = s[0], m1 = s[1], m2 = s[2], m3 = s[3];
#pragma unroll
            for (int i = 4; i < kHalf; i += 8) {
                m0 = ptx::max3(m0, s[i + 0], s[i + 1]);
                m1 = ptx::max3(m1, s[i + 2], s[i + 3]);
                if (i + 4 < kHalf) {
                    m2 = ptx::max3(m2, s[i + 4], s[i + 5]);
                    m3 = ptx::max3(m3, s[i + 6], s[i + 7]);
                }
            }
            m0 = ptx::max3(fmaxf(m0, m1), m2, m3);
            const uint32_t place = static_cast<uint32_t>(j & 1) * (2 * kTile * 4);
            ptx::st_shared_f32(max_own + place, m0);
            // P and O are free once the MMAs of the previous key tile are complete: at d = 64, and where the units take turns, by now, as a
            // rule, and the wait runs beside the other half's; two query tiles at d = 128 take longer than the maxima (976 -> 1022 us).
            auto products_done = [&]() {
                return static_cast<bool>(__all_sync(0xffffffffu, wait_in_place(&bars->p_free[q], (static_cast<uint32_t>(j) & 1u) ^ 1u, abort_flag, kSitePFree)));
            };
            if constexpr (turns) {
                ok = products_done();
                take_turn(j);
                if (!ok) {
                    pass_turn(j);
                    continue;
                }
            } else {
                __syncwarp();
                ptx::mbar_arrive_if(bar_of(offsetof(Barriers, max_full), q * 4 + quarter), lane0);
                ok = __all_sync(0xffffffffu, wait_in_place(&bars->max_full[q][quarter], static_cast<uint32_t>(j) & 1u, abort_flag, kSiteMaxFull));
                if (!ok) continue;
            }
            smax = ptx::max3(smax, m0, ptx::ld_shared_f32(max_other + place));
            const float mb_cand = fmaxf(smax * c2, -3.0e38f);
            const bool move = j == 0 || mb_cand - mb > kLazy;
            if constexpr (!turns) {
                ok = products_done();
                if (!ok) continue;
            }
            ptx::tc_fence_after_sync();
            uint32_t w[16];  // 32 keys of P on their way to tensor memory
            if (j == 0) {
                mb = mb_cand;
            } else if (__any_sync(0xffffffffu, move)) {
                // rescale this thread's part of O's row and l to the new offset (factor 1 for the rows of the warp
                // that do not move; the other thread of the row takes the same decision)
                const float alpha = move ? ptx::ex2_approx(mb - mb_cand) : 1.0f;
                if (move) mb = mb_cand;
                l *= alpha;
                ptx::tc_fence_after_sync();
#pragma unroll 1
                for (int c = 0; c < D / 2; c += 8) {  // 8 columns at a time: the row of scores stays in registers
                    uint32_t r[8];
                    ptx::tmem_ld_32x32b_x8(o_own + static_cast<uint32_t>(c), r);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
                    ptx::tmem_st_32x32b_x8(o_own + static_cast<uint32_t>(c), r);
                }
                ptx::tmem_wait_st();
            }
            // ---- weights: p = 2^(c2 s - mb) (below 2^8), row sum, bf16, into tensor memory ----
            const uint64_t nmb2 = ptx::pack2(-mb, -mb);
            uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
            for (int g = 0; g < kHalf / 8; ++g) {  // 8 keys = one 16-byte piece of the row
                float p[8];
#pragma unroll
                for (int i = 0; i < 8; i += 2) {
                    float x0, x1;
                    ptx::unpack2(ptx::fma2(ptx::pack2(s[g * 8 + i], s[g * 8 + i + 1]), c2c2, nmb2), x0, x1);
                    p[i] = ptx::ex2_approx(x0);
                    p[i + 1] = ptx::ex2_approx(x1);
                    if (valid < kTile) {  // columns beyond N: weight zero
                        p[i] = (half * kHalf + g * 8 + i < valid) ? p[i] : 0.0f;
                        p[i + 1] = (half * kHalf + g * 8 + i + 1 < valid) ? p[i + 1] : 0.0f;
                    }
                    acc[(i >> 1) & 3] = ptx::add2(acc[(i >> 1) & 3], ptx::pack2(p[i], p[i + 1]));
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) w[(g & 3) * 4 + i] = ptx::pack_bf16x2(p[2 * i], p[2 * i + 1]);
                if (g == kPassAt) pass_turn(j);
                if ((g & 3) == 3) ptx::tmem_st_32x32b_x16(p_own + static_cast<uint32_t>((g >> 2) * 16), w);
            }
            float a0, a1, a2, a3;
            ptx::unpack2(ptx::add2(acc[0], acc[1]), a0, a1);
            ptx::unpack2(ptx::add2(acc[2], acc[3]), a2, a3);
            l += (a0 + a1) + (a2 + a3);
            ptx::tmem_wait_st();
            ptx::tc_fence_before_sync();  // orders P in tensor memory and the rescale of O before the MMAs that use them
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&bars->p_full[q]);
        }

        // ---- epilogue: O / l -> bf16 -> the query tile's shared memory -> TMA stores ----
        if (split || my_steps > 0) {  // (split: each unit has a step)
            // Two units of one query tile each finish alone.  Two units of the same query tile meet here: the four threads of a
            // row take D / 4 columns each of 2^(mb_0 - mb) O_0 + 2^(mb_1 - mb) O_1.
            const int u = split ? 0 : q;  // the barriers and the query tile this epilogue uses
            const float* peer = reinterpret_cast<const float*>(smem + L::kStatOff) + (q ^ 1) * kUnitStats;
            const float *l_peer = peer + row, *mb_peer = peer + 2 * kTile + row;  // split: the other unit's sums (of both halves) and offset
            if (ok) ok = warp_wait(bar_of(offsetof(Barriers, o_full), q), 0, abort_flag, kSiteOFull);
            if (ok && split) ok = warp_wait(bar_of(offsetof(Barriers, o_full), q ^ 1), 0, abort_flag, kSiteOFull);
            if (ok) {
                stats[half * kTile + row] = l;  // (the maxima have all been read: the last product has them behind it)
                if (half == 0) stats[2 * kTile + row] = mb;
                __syncwarp();
                ptx::mbar_arrive_if(bar_of(offsetof(Barriers, l_full), u), lane0);
                ok = warp_wait(bar_of(offsetof(Barriers, l_full), u), 0, abort_flag, kSiteLFull);
            }
            if constexpr (M == kCluster) {
                // The CTAs of a cluster have worked on other key tiles of the same query tile.  Each sends its rows' (offset, sum) to all; with
                // them every thread knows its row's global ones, scales its part of O and sends it to the CTA that owns the row (128 / G
                // rows each); after the cluster's barrier the owners add the G parts, in the order of the CTAs, and write O.  The pairs complete
                // bytes on their readers' mbarriers: with a barrier of the cluster there too 2 x 1798, d = 128 took 13.3 us (now 12.9), 1 x 2500
                // 14.5 (14.25); the parts by such stores were slower (1 x 2500, d = 128 14.5 -> 15.4 us).
                const int my_rows = kTile / G;
                const float l_own = ok ? l + stats[(half ^ 1) * kTile + row] : 1.0f;
                const float mb_other = ok ? *mb_peer : 0.0f;
                if (ok && q == 0 && half == 0) {
                    const float top = fmaxf(mb, mb_other);
                    const uint64_t pair = ptx::pack2(top, l_own * ptx::ex2_approx(mb - top) + (l_peer[0] + l_peer[kTile]) * ptx::ex2_approx(mb_other - top));
                    for (int g = 0; g < G; ++g)
                        ptx::st_async_b64(ptx::map_to_cta(ptx::smem_u32(smem + L::kPairOff + (rank * kTile + row) * 8), static_cast<uint32_t>(g)), pair,
                                          ptx::map_to_cta(ptx::smem_u32(&bars->pairs_in), static_cast<uint32_t>(g)));
                }
                __syncwarp();
                if (ok) ok = warp_wait(bar_of(offsetof(Barriers, pairs_in), 0), 0, abort_flag, kSitePairsIn);
                if (ok) {
                    // (every CTA has sent its pairs behind its last product: the rings of all are free)
                    const float2* pairs = reinterpret_cast<const float2*>(smem + L::kPairOff) + row;
                    float2 pair[kMaxCluster];
                    float top = -3.0e38f, sum = 0.0f;
#pragma unroll
                    for (int g = 0; g < kMaxCluster; ++g) {
                        pair[g] = pairs[(g < G ? g : 0) * kTile];
                        top = fmaxf(top, pair[g].x);
                    }
#pragma unroll
                    for (int g = 0; g < kMaxCluster; ++g) sum += g < G ? pair[g].y * ptx::ex2_approx(pair[g].x - top) : 0.0f;
                    const float inv = 1.0f / sum;
                    const float f_own = ptx::ex2_approx(mb - top) * inv, f_other = ptx::ex2_approx(mb_other - top) * inv;
                    ptx::tc_fence_after_sync();
                    const uint32_t o_unit = t_quarter + L::o_col(q);
                    const uint32_t o_peer = t_quarter + L::o_col(q ^ 1);
                    // float [G CTAs][128 / G rows][D], 16-byte pieces XOR-swizzled by row
                    const uint32_t owner = static_cast<uint32_t>(row / my_rows);
                    const uint32_t dst = ptx::map_to_cta(ptx::smem_u32(smem + L::kKOff) + static_cast<uint32_t>((rank * my_rows + row % my_rows) * D * 4), owner);
                    const int col0 = (q * 2 + half) * (D / 4);
#pragma unroll 1
                    for (int c = col0; c < col0 + D / 4; c += 16) {
                        uint32_t o[16], r[16];
                        ptx::tmem_ld_32x32b_x16(o_unit + static_cast<uint32_t>(c), o);
                        ptx::tmem_ld_32x32b_x16(o_peer + static_cast<uint32_t>(c), r);
                        ptx::tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float v[4];
#pragma unroll
                            for (int x = 0; x < 4; ++x)
                                v[x] = fmaf(__uint_as_float(r[4 * i + x]), f_other, __uint_as_float(o[4 * i + x]) * f_own);
                            ptx::st_cluster_v4(dst + (((static_cast<uint32_t>(c) >> 2) + static_cast<uint32_t>(i)) ^ static_cast<uint32_t>(lane & 7)) * 16u,
                                               v[0], v[1], v[2], v[3]);
                        }
                    }
                }
                __syncwarp();
                ptx::cluster_arrive_release();
                ptx::cluster_wait_acquire();
                if (ok) {
                    for (int idx = static_cast<int>(threadIdx.x); idx < my_rows * (D / 8); idx += kSmWarps * 32) {
                        const int r = idx / (D / 8), piece = idx % (D / 8);  // 8 columns of row r of this CTA's
                        const int at = row0 + rank * my_rows + r;
                        if (at >= N) continue;
                        float v[8] = {};
                        for (int g = 0; g < G; ++g) {
                            const float4* src = reinterpret_cast<const float4*>(smem + L::kKOff) + (g * my_rows + r) * (D / 4);
                            const float4 a = src[(2 * piece) ^ (r & 7)], b = src[(2 * piece + 1) ^ (r & 7)];
                            v[0] += a.x, v[1] += a.y, v[2] += a.z, v[3] += a.w;
                            v[4] += b.x, v[5] += b.y, v[6] += b.z, v[7] += b.w;
                        }
                        uint4 out;
                        out.x = ptx::pack_bf16x2(v[0], v[1]);
                        out.y = ptx::pack_bf16x2(v[2], v[3]);
                        out.z = ptx::pack_bf16x2(v[4], v[5]);
                        out.w = ptx::pack_bf16x2(v[6], v[7]);
                        reinterpret_cast<uint4*>(O + (static_cast<size_t>(bh) * N + at) * D)[piece] = out;
                    }
                }
            } else if (ok) {
                float f_own, f_other = 0.0f;
                const float l_own = l + stats[(half ^ 1) * kTile + row];
                if (split) {
                    const float mb_other = *mb_peer;
                    const float top = fmaxf(mb, mb_other);
                    f_own = ptx::ex2_approx(mb - top);
                    f_other = ptx::ex2_approx(mb_other - top);
                    const float inv = 1.0f / (l_own * f_own + (l_peer[0] + l_peer[kTile]) * f_other);
                    f_own *= inv;
                    f_other *= inv;
                } else {
                    f_own = 1.0f / l_own;
                }
                ptx::tc_fence_after_sync();
                const int cols = split ? D / 4 : D / 2;
                const int col0 = split ? (q * 2 + half) * (D / 4) : half * (D / 2);
                const uint32_t o_unit = t_quarter + L::o_col(q);
                const uint32_t o_peer = t_quarter + L::o_col(q ^ 1);
                const uint32_t dst_row = ptx::smem_u32(smem + L::kQOff + u * L::kTileBytes) + static_cast<uint32_t>(row * 128);
#pragma unroll 1
                for (int c = col0; c < col0 + cols; c += 16) {
                    uint32_t o[16];
                    ptx::tmem_ld_32x32b_x16(o_unit + static_cast<uint32_t>(c), o);
                    ptx::tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f_own);
                    if (split) {
                        uint32_t r[16];
                        ptx::tmem_ld_32x32b_x16(o_peer + static_cast<uint32_t>(c), r);
                        ptx::tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(fmaf(__uint_as_float(r[i]), f_other, __uint_as_float(o[i])));
                    }
                    const uint32_t dst = dst_row + static_cast<uint32_t>((c >> 6) * L::kAtomBytes);
                    const uint32_t piece = static_cast<uint32_t>((c & 63) >> 3);
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        uint32_t w[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            w[i] = ptx::pack_bf16x2(__uint_as_float(o[g * 8 + 2 * i]), __uint_as_float(o[g * 8 + 2 * i + 1]));
                        ptx::st_shared_v4(dst + (((piece + static_cast<uint32_t>(g)) ^ sw) << 4), w[0], w[1], w[2], w[3]);
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (quarter == 0 && half == 0 && q == u) {
                    ok = warp_wait(bar_of(offsetof(Barriers, out_filled), u), 0, abort_flag, kSiteOutFilled);
                    if (ok && lane == 0) {
                        for (int a = 0; a < L::kAtoms; ++a)
                            ptx::tma_store_3d(&tm_o, ptx::smem_u32(smem + L::kQOff + u * L::kTileBytes + a * L::kAtomBytes), a * 64,
                                              row0 + u * kTile, bh, ptx::policy_evict_first());
                        ptx::bulk_commit_group();
                        ptx::bulk_wait_group<0>();
                    }
                } else {
                    ptx::mbar_arrive_if(bar_of(offsetof(Barriers, out_filled), u), lane0);
                }
            }
        }
    }

    if constexpr (M == kCluster) {
        if (warp >= kSmWarps) {  // the Softmax warps' barrier, behind which no CTA writes into a peer
            __syncwarp();
            ptx::cluster_arrive_release();
            ptx::cluster_wait_acquire();
        }
    }
    // ---- teardown: every role falls through to here, also after a wait gave up ----
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {
        if constexpr (M == kCluster) wait_for_late_stores();
        // Unwinding: let the copies already in flight land before shared memory is released.
        if (warp == kProducer && lane == 0) {
            const long long t0 = clock64();
            for (int it = loads > kStages ? loads - kStages : 0; it < loads; ++it)
                while (!ptx::mbar_try_wait(&bars->k_full[it % kStages], static_cast<uint32_t>(it / kStages) & 1u) &&
                       clock64() - t0 < kWaitLimitCycles / 8) {
                }
            while (!ptx::mbar_try_wait(&bars->q_full, 0) && clock64() - t0 < kWaitLimitCycles / 8) {
            }
        }
    }
    if (warp == kMma) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc(tmem_base, kTmemCols);
    }
}

}  // namespace av1
}  // namespace attnw
