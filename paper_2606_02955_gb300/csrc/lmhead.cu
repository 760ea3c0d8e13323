// lmhead.cu -- step a1 fused with the LM head that produces the logits.  The logits of a
// masked position are x = W h (h its final hidden state [H], W the vocabulary projection
// [V, H]); instead of writing B*L*V logits and reading them back, a tcgen05 GEMM reduces
// each 128-row x BN-column accumulator tile (BN = 256 or 208 vocabulary entries) in its
// epilogue to one (max, sum of exp, first argmax) partial per row, straight from tensor
// memory.
//
// Launch sequence on one stream (all rows of one step), chained by programmatic dependent
// launches:
//   1. pack_rows_kernel      the masked rows' indices, their count and their hidden states,
//                            packed [R, H] (TMA-friendly); two kernels, compact_rows and
//                            gather_rows, before the pair GEMM
//   2. lmhead_gemm_kernel    persistent tcgen05 GEMM: warp 0 issues TMA loads into a ring of
//                            stages, warp 1 issues tcgen05.mma into one of two TMEM
//                            accumulators, warps 2-5 reduce (or store) the other one; solo
//                            or CTA-pair (cta_group::2) variants
//      lmhead_slab_kernel    (at most 32 rows) the operands swapped, W as the M = 128 side:
//                            each CTA streams one vocabulary slab, one partial per row
//      lmhead_wide_kernel    (up to 1536 or 4096 rows) the operands swapped on a CTA pair, W as the
//                            M = 256 side and up to 256 (or 320) rows as N
//   3. combine_rows_kernel   four warps per row fold its tile (or slab) partials in a fixed
//                            order
//   4. profile_select        steps a2-a5 on the confidences (profile_select.cu)
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <mutex>
#include <string>

#include "fdllm.h"
#include "fdllm_internal.cuh"
#include "ptx.cuh"
#include "tcgen05.cuh"

namespace fdllm {
namespace {

constexpr int BM = 128;  // rows per tile (TMEM lanes)
constexpr int BK = 64;   // hidden elements per stage: one 128-byte swizzle row of bf16
constexpr int kABytes = BM * BK * 2;
constexpr int kThreads = 192;         // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue
constexpr uint32_t kAccStride = 256;  // TMEM columns between the two accumulators
constexpr uint32_t kTmemCols = 512;
constexpr size_t kBarrierBytes = 256;
constexpr size_t kRingBudget = 220 * 1024;
// kStore: an epilogue warp's 32 x 32 block of logits on its way to memory, rows padded to 33 so
// that writing it by column and reading it by row are both free of bank conflicts.
constexpr int kStagePitch = 33;
constexpr int kStageWarpFloats = 32 * kStagePitch;

// How the CTAs of a cluster share a W tile.
enum Mode {
    kSolo = 0,       // one CTA per work item; it loads the whole W tile
    kPair = 2,       // 2-CTA pair MMA (tcgen05 cta_group::2, M = 256): each CTA holds its 128
                     // rows and half of the W tile; the even CTA issues the MMAs for both
    kSlab = 3,       // at most 32 rows: W as the M = 128 operand, each CTA a vocabulary slab
                     // (lmhead_slab_kernel)
    kWide = 4,       // W as the M = 256 operand of a CTA pair, the rows as its N
                     // (lmhead_wide_kernel)
};

// Vocabulary entries per tile (the MMA's N and the fp32 accumulator's width): 256, or 208,
// which splits LLaDA's V = 126464 into 608 = 4 x 152 tiles, whole waves over 152 SMs.  The
// stage count fills the ring budget: solo 4 x 48 KB at 256, 5 x 42 KB at 208; pair 6 x 32 KB
// at 256 (each CTA holds half the W tile).  Three pair stages of two K-blocks each were the
// faster ring while issuing a stage cost as much as its MMAs; with warp-uniform issue the finer
// ring is: 28 x 32 rows 410 against 431 us, 32 x 32 rows 422 against 425, 64 x 32 rows 785
// against 787.
enum Epilogue { kReduce = 0, kStore = 1 };

template <int BN_, int MODE, int EPI = kReduce>
struct TileCfg {
    static constexpr int BN = BN_;
    static constexpr int kBRows = MODE == kPair ? BN / 2 : BN;  // W rows held per CTA
    static constexpr int kBBytes = kBRows * BK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr size_t kStagingBytes = EPI == kStore ? 4 * kStageWarpFloats * 4 : 0;
    static constexpr int kFit = (int)((kRingBudget - kStagingBytes) / kStageBytes);
    static constexpr int kStages = kFit > 8 ? 8 : kFit;
    static constexpr size_t kSmemBytes =
        1024 + (size_t)kStages * kStageBytes + kBarrierBytes + kStagingBytes;
    static_assert(kSmemBytes <= 227 * 1024, "ring and staging");
    static_assert(BN % 16 == 0 && BN <= (int)kAccStride, "MMA N");
    static_assert((BN / 2) % 8 == 0, "halves of whole 8-row swizzle atoms");
};

struct GemmArgs {
    const int32_t *row_count;  // R, written by the packing
    const int32_t *row_ids;    // [R] global row (b * L + l) of each packed row
    int32_t V;
    int32_t n_tiles;           // partials per row: ceil(V / BN), or the slab variant's grid
    int32_t k_blocks;          // ceil(H / BK)
    int32_t slab_tiles;        // slab variant: vocabulary tiles, ceil(V / slab_h)
    int32_t slab_h;            // slab variant: W rows per tile (a multiple of 8, <= 128)
    int32_t wide_h;            // wide variant: W rows per CTA and tile (a multiple of 8, <= 128)
    int32_t w_tiles;           // wide variant: vocabulary tiles of a CTA pair, ceil(V / 2 wide_h)
    UnitPartial *partials;     // kReduce: [R][n_tiles]
    float *logits;             // kStore: [B * L][V] fp32, written at masked rows
    uint32_t *status;          // sticky device error bits
    bool pdl;                  // host side: launch as a programmatic dependent
};

// A bounded wait that also gives up as soon as another role of the CTA has given up.
__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity, uint32_t *status,
                                              volatile int *abort_flag)
{
    if (mbar_try_wait(bar, parity))
        return true;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity))
            return true;
        if ((it & 63u) == 0) {
            if (*abort_flag)
                return false;
            if (global_timer_ns() - t0 > kWaitLimitNs) {
                atomicOr(status, kDevStatTimeout);
                *abort_flag = 1;
                return false;
            }
        }
    }
}

// wait_or_abort by a converged warp, the same answer in every lane.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, uint32_t *status,
                                          volatile int *abort_flag)
{
    if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity)))
        return true;
    return __all_sync(0xFFFFFFFFu, wait_or_abort(bar, parity, status, abort_flag));
}

// Waits (bounded) for the last `filled` fills of a ring of `stages` stages whose next fill would
// be that of stage s in phase ph: one thread, before its CTA may exit.
__device__ __forceinline__ void drain_ring(uint64_t *full, int stages, int s, uint32_t ph,
                                           uint32_t filled, uint32_t *status)
{
    for (uint32_t i = 0; i < filled; ++i) {
        if (s == 0) {
            s = stages;
            ph ^= 1u;
        }
        --s;
        mbar_wait(&full[s], ph, status, kDrainLimitNs);
    }
}

// MODE kSolo: every CTA loads its own W tile.  kPair: the two CTAs of a cluster take row
// tiles 2j and 2j + 1 of the same vocabulary tile, which form one M = 256 MMA issued by the
// even CTA (tcgen05 cta_group::2):
// each CTA loads its 128 rows and half of the W tile into its own shared memory and
// signals the even CTA's stage barrier, so each CTA's shared memory supplies half the
// operand bytes per MMA; the accumulators live in both CTAs' tensor memory.
template <int EPI, int MODE, int BN_>
__global__ void __launch_bounds__(kThreads, 1)
    lmhead_gemm_kernel(const __grid_constant__ CUtensorMap map_h,
                       const __grid_constant__ CUtensorMap map_w, const GemmArgs a)
{
    using Cfg = TileCfg<BN_, MODE, EPI>;
    constexpr int CL = MODE == kSolo ? 1 : 2;
    constexpr bool PAIR = MODE == kPair;
    constexpr int BN = Cfg::BN, kStages = Cfg::kStages;
    constexpr int kBBytes = Cfg::kBBytes, kStageBytes = Cfg::kStageBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem;                      // kStages x [BM rows][128 B], swizzled
    uint8_t *sB = smem + kStages * kABytes;  // kStages x [kBRows rows][128 B]
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + kStages * kBBytes);
    uint64_t *full = bars;                  // TMA -> MMA, one per stage
    uint64_t *empty = bars + kStages;       // MMA -> TMA, one per stage
    uint64_t *tfull = bars + 2 * kStages;   // MMA -> epilogue, one per accumulator
    uint64_t *tempty = tfull + 2;           // epilogue -> MMA, one per accumulator
    uint64_t *done = tempty + 2;            // MMA thread: all its MMAs have completed
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    float *staging = reinterpret_cast<float *>(reinterpret_cast<uint8_t *>(bars) + kBarrierBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);  // released by the MMA issuer's commit
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], PAIR ? 8 : 4);  // one arrival per epilogue warp (of the pair)
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        fence_mbar_init();
        tc::prefetch_tensormap(&map_h);
        tc::prefetch_tensormap(&map_w);
    }
    if (warp == 1) {
        if (PAIR)
            tc::tmem_alloc_pair(tmem_slot, kTmemCols);
        else
            tc::tmem_alloc(tmem_slot, kTmemCols);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (CL > 1)
        tc::cluster_sync();  // the peer's barriers are initialised before any remote signal
    tc::fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    // A programmatic dependent of the packing kernel: everything above overlapped it;
    // the packed rows and their count are read only past this wait.
    pdl_wait();

    const int rank = CL > 1 ? (int)tc::cluster_ctarank() : 0;
    const int64_t first = CL > 1 ? (int64_t)tc::cluster_id_x() : (int64_t)blockIdx.x;
    const int64_t stride = CL > 1 ? (int64_t)tc::cluster_count_x() : (int64_t)gridDim.x;
    // An epilogue warp hands an accumulator back to the MMA issuer (in a pair, the even
    // CTA's barrier counts the warps of both CTAs).
    auto release_acc = [](uint64_t *bar, int rk) {
        if (PAIR && rk != 0)
            tc::mbar_arrive_remote(tc::map_to_rank(bar, 0));
        else
            mbar_arrive(bar);
    };
    const int R = __shfl_sync(0xFFFFFFFFu, *a.row_count, 0);
    const int num_m = (R + BM - 1) / BM;
    const int num_mc = (num_m + CL - 1) / CL;  // row-tile groups, one per cluster
    const int64_t total = (int64_t)num_mc * a.n_tiles;
    // Work item t covers packed rows [m*BM, +BM) with m = (t % num_mc) * CL + rank, and
    // vocabulary [n*BN, +BN) with n = t / num_mc: row tiles fastest, so the CTAs working at
    // the same time share few W tiles (read from HBM once, then from L2).  With CL = 2 and
    // an odd number of row tiles, the last rank-1 CTA computes a tile of rows >= R (zero or
    // stale inputs) that its epilogue skips.

    // Warps 0 and 1 run whole, one elected lane issuing: loop state and operand addresses then
    // stay warp-uniform, which the issuing instructions need them to be.  Against loops under
    // `lane == 0` (and the pair's stages as they were): 32 x 32 rows 434 against 439 us, 64 x 32
    // 800 against 807, the slab variant at 24 rows 154.3 against 156.8.
    if (warp == 0) {
        // W tiles are marked first to evict: each is read from HBM once, and the other row
        // tiles that share it (consecutive work items) read it from L2 right away.
        const uint64_t pol = make_evict_first_policy();
        int s = 0;
        uint32_t ph = 0, filled = 0;
        bool ok = true;
        for (int64_t t = first; ok && t < total; t += stride) {
            const int m = (int)(t % num_mc) * CL + rank, n = (int)(t / num_mc);
            for (int kb = 0; kb < a.k_blocks; ++kb) {
                if (!warp_wait(&empty[s], ph ^ 1u, a.status, abort_flag)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    if constexpr (PAIR) {
                        // Both CTAs' bytes complete on the even CTA's barrier, which it arms.
                        if (rank == 0)
                            mbar_arrive_expect_tx(&full[s], 2 * kStageBytes);
                        const uint32_t bar0 = tc::map_to_rank(&full[s], 0);
                        tc::tma_load_2d_pair(sA + s * kABytes, &map_h, kb * BK, m * BM, bar0);
                        tc::tma_load_2d_pair(sB + s * kBBytes, &map_w, kb * BK,
                                             n * BN + rank * (BN / 2), bar0);
                    } else {
                        mbar_arrive_expect_tx(&full[s], kStageBytes);
                        tc::tma_load_2d(sA + s * kABytes, &map_h, kb * BK, m * BM, &full[s]);
                        tc::tma_load_2d_hint(sB + s * kBBytes, &map_w, kb * BK, n * BN, &full[s],
                                             pol);
                    }
                }
                filled = min(filled + 1, (uint32_t)kStages);
                if (++s == kStages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        // No copy of this CTA may still be in flight when it exits (in a pair, the even
        // CTA's barriers count both CTAs' copies, and the odd CTA leaves only after it,
        // at the final cluster barrier).
        if ((!PAIR || rank == 0) && elect_one())
            drain_ring(full, kStages, s, ph, filled, a.status);
        __syncwarp();
    } else if (warp == 1) {
        if (!PAIR || rank == 0) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(PAIR ? 2 * BM : BM, BN);
            int s = 0;
            uint32_t ph = 0;
            bool ok = true;
            int i = 0;
            for (int64_t t = first; ok && t < total; t += stride, ++i) {
                const int acc = i & 1;
                const uint32_t aph = (uint32_t)(i >> 1) & 1u;
                if (!warp_wait(&tempty[acc], aph ^ 1u, a.status, abort_flag))
                    break;
                tc::fence_after_sync();
                const uint32_t d = tmem_base + (uint32_t)acc * kAccStride;
                for (int kb = 0; kb < a.k_blocks; ++kb) {
                    if (!warp_wait(&full[s], ph, a.status, abort_flag)) {
                        ok = false;
                        break;
                    }
                    tc::fence_after_sync();
                    if (elect_one()) {
                        const uint64_t ad = tc::sw128_kmajor_desc(sA + s * kABytes);
                        const uint64_t bd = tc::sw128_kmajor_desc(sB + s * kBBytes);
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {  // K = 16 per MMA: +32 B in the row
                            if constexpr (PAIR)
                                tc::mma_bf16_pair(d, ad + 2u * k, bd + 2u * k, idesc,
                                                  (kb | k) != 0);
                            else
                                tc::mma_bf16(d, ad + 2u * k, bd + 2u * k, idesc, (kb | k) != 0);
                        }
                        // The stage is free once these MMAs have read it (in a pair, in both
                        // CTAs: each refills its own half of the pair's operands).
                        if constexpr (PAIR)
                            tc::commit_pair_multicast(&empty[s]);
                        else
                            tc::commit(&empty[s]);
                    }
                    if (++s == kStages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                if (ok && elect_one()) {
                    if constexpr (PAIR)
                        tc::commit_pair_multicast(&tfull[acc]);  // both CTAs' accumulators
                    else
                        tc::commit(&tfull[acc]);
                }
            }
            // Tensor memory is freed below only after every MMA issued here has completed.
            __syncwarp();
            if (elect_one()) {
                if constexpr (PAIR)
                    tc::commit_pair_multicast(done);  // the odd CTA's copy is never waited on
                else
                    tc::commit(done);
                mbar_wait(done, 0, a.status, kDrainLimitNs);
            }
        }
        __syncwarp();
    } else {
        // Epilogue: warp w reads TMEM lanes [32 (w % 4), +32): thread = one row of the tile.
        const int quarter = warp & 3;
        const int row_in_tile = quarter * 32 + lane;
        int i = 0;
        for (int64_t t = first; t < total; t += stride, ++i) {
            const int acc = i & 1;
            const uint32_t aph = (uint32_t)(i >> 1) & 1u;
            const int m = (int)(t % num_mc) * CL + rank, n = (int)(t / num_mc);
            // Every lane waits; the warp leaves together if any lane gave up, so that the
            // warp-collective tensor-memory loads below are always executed by all lanes.
            const bool ok = wait_or_abort(&tfull[acc], aph, a.status, abort_flag);
            if (!__all_sync(0xFFFFFFFFu, ok))
                break;
            tc::fence_after_sync();
            const uint32_t taddr =
                tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * kAccStride;
            const int r = m * BM + row_in_tile;
            const int col0 = n * BN;
            float v[32];
            if (EPI == kReduce) {
                // Pass 1: max and its first column; NaN is tracked apart (fmax would drop it).
                float M = -__int_as_float(0x7F800000);
                uint32_t idx = kNoIdx;
                bool nan = false;
#pragma unroll 1
                for (int c = 0; c < (BN + 31) / 32; ++c) {
                    tc::tmem_ld_32cols(taddr + c * 32, v);  // columns >= BN: not this tile
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int col = col0 + c * 32 + j;
                        if (c * 32 + j < BN && col < a.V) {
                            nan |= v[j] != v[j];
                            if (v[j] > M) {
                                M = v[j];
                                idx = (uint32_t)col;
                            }
                        }
                    }
                }
                // Pass 2: sum of exp(x - M) = 2^(x sc - M2), four partial sums, with the
                // scale sc and reference M2 of rebase_scaled (sc = 1 and M2 = M for |M| at or
                // beyond kBigRef, where only x == M contributes).
                const bool big = !(fabsf(M) < kBigRef);
                const float sc = big ? 1.0f : kLog2e;
                const float M2 = big ? M : M * kLog2e;
                float S4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
                for (int c = 0; c < (BN + 31) / 32; ++c) {
                    tc::tmem_ld_32cols(taddr + c * 32, v);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const int col = col0 + c * 32 + j;
                        if (c * 32 + j < BN && col < a.V)
                            S4[j & 3] += ex2_mufu(fmaf(v[j], sc, -M2));
                    }
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0)
                    release_acc(&tempty[acc], rank);
                if (r < R) {
                    UnitPartial p;
                    p.M = nan ? __int_as_float(0x7FC00000) : M;
                    // relative to M exactly; a tile with no finite logit adds exactly 0
                    p.S = M == -INFINITY
                              ? 0.0f
                              : rebase_scaled((S4[0] + S4[1]) + (S4[2] + S4[3]), sc, M2, M);
                    p.idx = idx;
                    p.pad = 0;
                    a.partials[(int64_t)r * a.n_tiles + n] = p;
                }
            } else {
                // A lane holds 32 columns of its own row, so storing from the registers would
                // touch 32 rows per instruction: 122 us for 192 rows of 50001 logits at
                // H = 2048.  The block turns in shared memory and leaves row by row, 128
                // consecutive bytes per instruction: 61 us.
                float *block = staging + quarter * kStageWarpFloats;
                const int row = r < R ? a.row_ids[r] : -1;
                const int live = min(R - (m * BM + quarter * 32), 32);  // the warp's rows < R
#pragma unroll 1
                for (int c = 0; c < (BN + 31) / 32; ++c) {
                    tc::tmem_ld_32cols(taddr + c * 32, v);
                    __syncwarp();  // the block's last rows have been read
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        block[lane * kStagePitch + j] = v[j];
                    __syncwarp();
                    const int col = col0 + c * 32 + lane;
                    const bool in = c * 32 + lane < BN && col < a.V;
#pragma unroll 4
                    for (int i = 0; i < live; ++i) {
                        const int64_t row_i = __shfl_sync(0xFFFFFFFFu, row, i);
                        if (in)
                            a.logits[row_i * a.V + col] = block[i * kStagePitch + lane];
                    }
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0)
                    release_acc(&tempty[acc], rank);
            }
        }
    }
    if (threadIdx.x == 0)
        pdl_launch_dependents();  // the row combination may start launching
    __syncthreads();
    if (PAIR)
        tc::cluster_sync();  // both CTAs are done with the pair's tensor memory
    if (warp == 1) {
        __syncwarp();
        tc::fence_after_sync();
        if (PAIR)
            tc::tmem_dealloc_pair(tmem_base, kTmemCols);
        else
            tc::tmem_dealloc(tmem_base, kTmemCols);
    }
    if (CL > 1)
        tc::cluster_sync();  // no CTA leaves while its peer may still write into it
}

// ----------------------------------------------------------------------------- slab variant
// For at most kSlabRows masked rows the operands swap roles: W is the MMA's A operand (M =
// 128 TMEM lanes, lane = vocabulary entry) and the packed rows are its B operand (N = 32,
// TMEM column = row).  The vocabulary is cut into tiles of h entries (one TMA box of h W
// rows, h a multiple of 8 up to 128, chosen by the host so that the busiest CTA streams as
// few W rows as possible: LLaDA's V = 126464 is 1216 tiles of 104, eight per SM on 152
// SMs); CTA c of P owns the tiles c, c + P, c + 2P, ..., so the CTAs read W in a window that
// moves through it.  The MMA always spans 128 lanes; lanes h..127 hold sums of stale shared
// memory that the epilogue skips.  The padded row tile costs 4 KB per K-block instead of
// 16 KB.  A stage holds two K-blocks (two W boxes and two row boxes), five stages in all
// (130 KB of W at h = 104 in flight per SM): per-copy overhead, not the bytes in flight,
// limits how fast W streams here, and two blocks per stage beat one, three or four.  Each
// epilogue thread keeps, for each of its 16 rows, a running maximum, sum of exp relative to it and
// first index over its own entry of each tile; after the last tile the 128 entries' states
// are folded per row (a transposing butterfly in each warp, then the four warps in order)
// into one partial per (row, CTA).
constexpr int kSlabRows = 32;
constexpr int kSlabABytes = BM * BK * 2;                 // 128 lanes; a tile fills h rows
constexpr int kSlabBBytes = kSlabRows * BK * 2;
constexpr int kSlabKB = 2;                               // K-blocks of BK per stage
constexpr int kSlabStages = 5;
constexpr int kSlabAccs = 4;                             // accumulators of 32 columns
constexpr uint32_t kSlabTmemCols = 128;
// Two epilogue warps per TMEM lane quarter, 16 rows each: the last tile's reduction and the fold
// over the entries are the kernel's tail.  Whole fdllm_lmhead_confidence pass, one warp of 32 rows
// against two of 16: 24 rows, H = 1024, 20000 entries 13.9 -> 12.9 us, 8000 10.6 -> 10.2, H = 2048,
// 65000 46.2 -> 45.4, LLaDA's head 151.9 -> 151.2.
constexpr int kSlabWarps = 8;
constexpr int kSlabWarpRows = kSlabRows / (kSlabWarps / 4);
constexpr int kSlabThreads = 64 + kSlabWarps * 32;
constexpr size_t kSlabSmemBytes =
    1024 + (size_t)kSlabStages * kSlabKB * (kSlabABytes + kSlabBBytes) + kBarrierBytes;
static_assert(kSlabSmemBytes <= 227 * 1024, "slab ring");
static_assert((2 * kSlabStages + 2 * kSlabAccs + 1) * 8 + 8 <= (int)kBarrierBytes, "barriers");

// Two (max, sum relative to it, first index) states of one row -> one.  NaN logits reach
// only S (they never raise the max), which then stays NaN.
__device__ __forceinline__ void fold_state(float &M, float &S, uint32_t &I, float M2, float S2,
                                           uint32_t I2)
{
    const float Mn = fmaxf(M, M2);
    S = rebase(S, M, Mn) + rebase(S2, M2, Mn);
    const uint32_t i1 = M == Mn ? I : kNoIdx, i2 = M2 == Mn ? I2 : kNoIdx;
    I = i1 < i2 ? i1 : i2;
    M = Mn;
}

template <int EPI>
__global__ void __launch_bounds__(kSlabThreads, 1)
    lmhead_slab_kernel(const __grid_constant__ CUtensorMap map_h,
                       const __grid_constant__ CUtensorMap map_w, const GemmArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ float s_M[4][kSlabRows], s_S[4][kSlabRows];
    __shared__ uint32_t s_I[4][kSlabRows];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // kSlabStages x kSlabKB x [128 W rows][128 B], then kSlabStages x kSlabKB x [32 rows][128 B]
    uint8_t *sA = smem;
    uint8_t *sB = smem + kSlabStages * kSlabKB * kSlabABytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + kSlabStages * kSlabKB * kSlabBBytes);
    uint64_t *full = bars;
    uint64_t *empty = bars + kSlabStages;
    uint64_t *tfull = bars + 2 * kSlabStages;
    uint64_t *tempty = tfull + kSlabAccs;
    uint64_t *done = tempty + kSlabAccs;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlabStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < kSlabAccs; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], kSlabWarps);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        fence_mbar_init();
        tc::prefetch_tensormap(&map_h);
        tc::prefetch_tensormap(&map_w);
    }
    if (warp == 1)
        tc::tmem_alloc(tmem_slot, kSlabTmemCols);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    pdl_wait();  // the packed rows and their count are complete

    const int R = __shfl_sync(0xFFFFFFFFu, *a.row_count, 0);  // <= kSlabRows: the host's choice
    const int64_t NT = a.slab_tiles, P = gridDim.x, c = blockIdx.x;
    const int h = a.slab_h;
    const int n_t = R > 0 && c < NT ? (int)((NT - c + P - 1) / P) : 0;  // tiles of this CTA

    if (warp == 0) {  // warps 0 and 1 whole, one elected lane issuing, as in the tile GEMM
        const uint64_t pol = make_evict_first_policy();  // W is read once
        int s = 0;
        uint32_t ph = 0, filled = 0;
        bool ok = true;
        // a box's bytes count in full, the part beyond V zero-filled
        // (K-blocks past H, in the last stage when k_blocks is odd, are zero-filled and
        // count in full too)
        const uint32_t bytes = kSlabKB * ((uint32_t)(h * BK * 2) + kSlabBBytes);
        for (int t = 0; ok && t < n_t; ++t) {
            const int64_t T = c + (int64_t)t * P;
            for (int kb = 0; kb < a.k_blocks; kb += kSlabKB) {
                if (!warp_wait(&empty[s], ph ^ 1u, a.status, abort_flag)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    mbar_arrive_expect_tx(&full[s], bytes);
#pragma unroll
                    for (int q = 0; q < kSlabKB; ++q)
                        tc::tma_load_2d_hint(sA + (s * kSlabKB + q) * kSlabABytes, &map_w,
                                             (kb + q) * BK, (int32_t)(T * h), &full[s], pol);
#pragma unroll
                    for (int q = 0; q < kSlabKB; ++q)
                        tc::tma_load_2d(sB + (s * kSlabKB + q) * kSlabBBytes, &map_h, (kb + q) * BK,
                                        0, &full[s]);
                }
                filled = min(filled + 1, (uint32_t)kSlabStages);
                if (++s == kSlabStages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        if (elect_one())  // none of this CTA's copies in flight at exit
            drain_ring(full, kSlabStages, s, ph, filled, a.status);
        __syncwarp();
    } else if (warp == 1) {
        constexpr uint32_t idesc = tc::idesc_bf16_f32(BM, kSlabRows);
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int t = 0; ok && t < n_t; ++t) {
            const int acc = t % kSlabAccs;
            const uint32_t aph = (uint32_t)(t / kSlabAccs) & 1u;
            if (!warp_wait(&tempty[acc], aph ^ 1u, a.status, abort_flag))
                break;
            tc::fence_after_sync();
            const uint32_t d = tmem_base + (uint32_t)(acc * kSlabRows);
            for (int kb = 0; kb < a.k_blocks; kb += kSlabKB) {
                if (!warp_wait(&full[s], ph, a.status, abort_flag)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                // Rows h..127 of the A stage are stale: those TMEM lanes hold
                // meaningless sums that the epilogue skips.
                if (elect_one()) {
#pragma unroll
                    for (int q = 0; q < kSlabKB; ++q) {
                        const uint64_t ad =
                            tc::sw128_kmajor_desc(sA + (s * kSlabKB + q) * kSlabABytes);
                        const uint64_t bd =
                            tc::sw128_kmajor_desc(sB + (s * kSlabKB + q) * kSlabBBytes);
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k)
                            tc::mma_bf16(d, ad + 2u * k, bd + 2u * k, idesc, (kb | q | k) != 0);
                    }
                    tc::commit(&empty[s]);
                }
                if (++s == kSlabStages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (ok && elect_one())
                tc::commit(&tfull[acc]);
        }
        __syncwarp();
        if (elect_one()) {
            tc::commit(done);
            mbar_wait(done, 0, a.status, kDrainLimitNs);
        }
        __syncwarp();
    } else {
        // Epilogue: warp w reads TMEM lanes [32 (w % 4), +32): thread = one vocabulary entry
        // of the tile, its columns = kSlabWarpRows of the rows, from row0 on.
        const int q = warp & 3, row0 = (warp - 2) / 4 * kSlabWarpRows;
        float M[kSlabWarpRows], S[kSlabWarpRows];
        uint32_t I[kSlabWarpRows];
#pragma unroll
        for (int r = 0; r < kSlabWarpRows; ++r) {
            M[r] = -__int_as_float(0x7F800000);
            S[r] = 0.0f;
            I[r] = kNoIdx;
        }
        bool aborted = false;
        for (int t = 0; t < n_t; ++t) {
            const int acc = t % kSlabAccs;
            const uint32_t aph = (uint32_t)(t / kSlabAccs) & 1u;
            const bool ok = wait_or_abort(&tfull[acc], aph, a.status, abort_flag);
            if (!__all_sync(0xFFFFFFFFu, ok)) {
                aborted = true;
                break;
            }
            tc::fence_after_sync();
            float v[kSlabWarpRows];
            tc::tmem_ld_16cols_async(tmem_base + ((uint32_t)(q * 32) << 16) +
                                         (uint32_t)(acc * kSlabRows + row0),
                                     v);
            tc::tmem_wait_ld();
            tc::tie_regs(v);
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&tempty[acc]);
            // lane q * 32 + lane of tile c + tP: vocabulary entry (c + tP) * h + q * 32 + lane
            const int in_tile = q * 32 + lane;
            const int64_t ent = (c + (int64_t)t * P) * h + in_tile;
            if (in_tile >= h || ent >= a.V)
                continue;
            if (EPI == kStore) {
#pragma unroll
                for (int r = 0; r < kSlabWarpRows; ++r)
                    if (row0 + r < R)
                        a.logits[(int64_t)a.row_ids[row0 + r] * a.V + ent] = v[r];
            } else {
#pragma unroll
                for (int r = 0; r < kSlabWarpRows; ++r) {
                    // exp(x - M) in the form (x - M) * log2e, exact at any magnitude; a
                    // larger x re-bases the sum; -inf adds nothing; NaN poisons S
                    const float x = v[r];
                    const bool up = x > M[r];
                    const float e = ex2_mufu((up ? M[r] - x : x - M[r]) * kLog2e);
                    S[r] = up ? fmaf(S[r], e, 1.0f) : (x == -INFINITY ? S[r] : S[r] + e);
                    I[r] = up ? (uint32_t)ent : I[r];
                    M[r] = up ? x : M[r];
                }
            }
        }
        if (EPI == kReduce) {
            // Transposing butterfly: at offset o each lane keeps the half of its remaining
            // row slots selected by its lane bit o and folds in the partner's values for them;
            // slot 0 ends as row row0 + lane % 16, folded over half of the warp's 32 entries, then
            // over both.
            const int mine = lane & (kSlabWarpRows - 1);
#pragma unroll
            for (int o = kSlabWarpRows / 2; o >= 1; o >>= 1) {
                const bool hi = (lane & o) != 0;
#pragma unroll
                for (int j = 0; j < o; ++j) {
                    const float sM = hi ? M[j] : M[j + o], sS = hi ? S[j] : S[j + o];
                    const uint32_t sI = hi ? I[j] : I[j + o];
                    float kM = hi ? M[j + o] : M[j], kS = hi ? S[j + o] : S[j];
                    uint32_t kI = hi ? I[j + o] : I[j];
                    const float rM = __shfl_xor_sync(0xFFFFFFFFu, sM, o);
                    const float rS = __shfl_xor_sync(0xFFFFFFFFu, sS, o);
                    const uint32_t rI = __shfl_xor_sync(0xFFFFFFFFu, sI, o);
                    fold_state(kM, kS, kI, rM, rS, rI);
                    M[j] = kM;
                    S[j] = kS;
                    I[j] = kI;
                }
            }
            fold_state(M[0], S[0], I[0], __shfl_xor_sync(0xFFFFFFFFu, M[0], kSlabWarpRows),
                       __shfl_xor_sync(0xFFFFFFFFu, S[0], kSlabWarpRows),
                       __shfl_xor_sync(0xFFFFFFFFu, I[0], kSlabWarpRows));
            if (lane < kSlabWarpRows) {
                s_M[q][row0 + mine] = M[0];
                s_S[q][row0 + mine] = S[0];
                s_I[q][row0 + mine] = I[0];
            }
            // every epilogue warp arrives exactly once, aborted or not
            asm volatile("bar.sync 1, %0;" ::"n"(kSlabWarps * 32) : "memory");
            if (warp == 4 && !aborted && !*abort_flag && lane < R) {
                float fM = s_M[0][lane], fS = s_S[0][lane];
                uint32_t fI = s_I[0][lane];
                for (int w = 1; w < 4; ++w)
                    fold_state(fM, fS, fI, s_M[w][lane], s_S[w][lane], s_I[w][lane]);
                UnitPartial p;
                p.M = fS != fS ? __int_as_float(0x7FC00000) : fM;
                p.S = fS;
                p.idx = fI;
                p.pad = 0;
                a.partials[(int64_t)lane * a.n_tiles + blockIdx.x] = p;
            }
        }
    }
    if (threadIdx.x == 0)
        pdl_launch_dependents();  // the row combination may start launching
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem_base, kSlabTmemCols);
    }
}

// ----------------------------------------------------------------------------- wide variant
// W is the M = 256 operand of a CTA pair (a tile of 2 h vocabulary entries, h <= 128 per CTA, lane
// = entry, see wide_height) and the packed rows are N, in blocks of up to 256 rows (one MMA group,
// two accumulators in turn) or, for 257 to 320 rows, one block of two groups that share every W
// stage (three accumulators).
// What bounds the solo variant at 2 to 6 row tiles is the 64 B/clock at which an SM receives from
// L2: its stage is 42 KB for 416 MMA cycles (101 B/clock wanted, 65 measured).
// Here a stage is (128 + N / 2) x 128 B for 2 N cycles: 75 B/clock at N = 192, 58 at 320, and no
// row tile is padded to 128.  LLaDA's head, 3/4 of B x 32 rows, whole fdllm_lmhead_confidence
// pass, this variant against the better of solo and pair: B = 3 (72 rows) 160 against 163 us,
// 8 165 against 190, 12 194 against 251, 16 244 against 261, 24 338 against 397, 28 376 against
// 405 (more rows at gemm_mode).
// Other cuts measured: 288 rows in two blocks 220, in two groups of 160 instead of 160 and 128
// 200 (back to back, at the power limit, 235 against 225), 381 rows in one block of two groups
// 245, 480 rows in one block 311 against 293 in two.
constexpr int kWideMaxGroup = 256;              // MMA columns per group
constexpr int kWideTwoGroups = 320;             // rows that still make one block, of two groups
// A few rows leave room for 12 and more stages, but W streams faster with fewer of its bytes in
// flight: of 4 x 32 rows 8 masked 161 us with 14 stages, 155.5 with 12, 154.2 with 11, 154.4 with
// 10, 157 with 8; 64 masked 159.5, 156.6, 157.2 and 160 (12, 11, 10, 8), 96 masked 157.8, 157.9,
// 158.3 and 161.3; H = 1024, 100000 entries, 8 masked 39.7, 39.1, 38.5 and 38.4.
constexpr int kWideMaxStages = 11;
constexpr int kWideWarps = 12;                  // epilogue warps, three per TMEM lane quarter
constexpr int kWideSplit = kWideWarps / 4;
constexpr int kWideThreads = 64 + kWideWarps * 32;
constexpr size_t kWideBarBytes = 512;
constexpr size_t kWideQuarters = (size_t)4 * kWideMaxGroup * (4 + 4 + 1);
constexpr size_t kWideSmemBytes = 227 * 1024;
constexpr size_t kWideFixed = kWideBarBytes + kWideQuarters;
static_assert((2 * kWideMaxStages + 2 * 4 + 1) * 8 + 8 <= (int)kWideBarBytes, "barriers");

// Tensor maps of the packed rows, box heights 16, 32, ..., 128: entry h / 16 - 1 loads half a
// group's rows.
constexpr int kWideMaps = kWideMaxGroup / 32;
struct WideRowMaps {
    CUtensorMap m[kWideMaps];
};

// How R rows are cut: n_blocks blocks of g rows, or one block of two groups of g and g1 rows, both
// multiples of 32 (what lies past R is padding), items (W tile, block) with the block fastest, so
// that the pairs sharing a W tile work on it at the same time.  `buffers` accumulators of g
// columns take turns.
struct WideCut {
    int n_blocks, groups, g, g1, buffers;
};

__device__ __forceinline__ WideCut wide_cut(int R)
{
    WideCut c;
    c.n_blocks = R > kWideTwoGroups ? (R + kWideMaxGroup - 1) / kWideMaxGroup : R > 0;
    const int per = c.n_blocks > 0 ? (R + c.n_blocks - 1) / c.n_blocks : 1;
    c.groups = per > kWideMaxGroup ? 2 : 1;
    c.g = ((per + c.groups - 1) / c.groups + 31) / 32 * 32;
    c.g1 = c.groups == 2 ? (per - c.g + 31) / 32 * 32 : 0;
    c.buffers = min(4, (int)kTmemCols / c.g);
    return c;
}

// What a CTA pair works on at a time: W tile n and the rows from row0 on, in one group of w0 or two
// of w0 and w1 columns.
struct WidePiece {
    int n, row0, w0, w1;
};

// The pieces of one CTA pair.  Whole rounds of items over the pairs first; if what is left then
// fills at most half of them, each leftover item goes to two pairs, one group or half of the one
// group each: halves of 96 and 64 columns (a group of 160) and up; no narrower group was tried.
// Whole fdllm_lmhead_confidence pass with one-group items left whole against halved: 200 rows, H =
// 4096, 20000 entries 49.5 -> 46.4 us, 65000 entries 98.7 -> 95.8, LLaDA's 169 -> 167; H = 1024,
// 20000 entries 200 rows 20.6 -> 19.5, 700 rows 32.9 -> 31.4; H = 2048, 8000 entries 200 rows 19.5
// -> 17.5.  In a group of 160: 144 rows, H = 1024, 20000 entries 19.3 -> 18.1, H = 4096, 25000
// entries 48.2 -> 47.5, LLaDA's 162.2 -> 161.8; 160 rows, H = 2048, 45000 entries 42.5 -> 41.6.
constexpr int kWideHalved = 160;

struct WideItems {
    const WideCut cut;
    // items of whole rounds, all items (B * L * V / 208 < 2^31 keeps them small), this pair
    int whole, total, pairs, pair;
    int first;  // columns of a leftover item's first part; 0: not cut

    __device__ __forceinline__ WideItems(const WideCut &c, int n_w_tiles, int pairs_, int pair_)
        : cut(c), total(n_w_tiles * c.n_blocks), pairs(pairs_), pair(pair_)
    {
        const int left = total % pairs;
        whole = total - left;
        first = 2 * left > pairs       ? 0
                : c.groups == 2        ? c.g
                : c.g >= kWideHalved   ? (c.g / 2 + 31) / 32 * 32
                                       : 0;
    }
    // The pair's i-th piece; false past the last.
    __device__ __forceinline__ bool piece(int i, WidePiece &p) const
    {
        int t = i * pairs + pair;
        p.w0 = cut.g;
        p.w1 = cut.g1;
        int off = 0;
        if (t >= whole) {
            if (i != whole / pairs)
                return false;
            if (first != 0) {
                t = whole + pair / 2;
                p.w0 = first;
                p.w1 = 0;
                if (pair & 1) {
                    off = first;
                    p.w0 = cut.g + cut.g1 - first;
                }
            }
            if (t >= total)
                return false;
        }
        p.n = t / cut.n_blocks;
        p.row0 = t % cut.n_blocks * cut.g + off;  // one block where there are two groups
        return true;
    }
};

// Folds the states (M, S relative to M, first index) of one column from two sets of entries. Either
// order gives the same bits.  -inf logits have S = 0; a NaN one leaves S NaN.
__device__ __forceinline__ void wide_fold(float &M, float &S, uint32_t &I, float M2, float S2,
                                          uint32_t I2)
{
    const bool up = M2 > M;
    const float hi = up ? M2 : M, lo = up ? M : M2;
    const float e = lo == -INFINITY ? 0.0f : ex2_mufu((lo - hi) * kLog2e);
    I = up ? I2 : (M2 == M ? min(I, I2) : I);
    S = fmaf(up ? S : S2, e, up ? S2 : S);
    M = hi;
}

// The column of a 32-column block whose state wide_reduce_block leaves in this lane.
__device__ __forceinline__ int wide_column(int lane)
{
    return (lane >> 3) * 8 + (lane & 3) * 2 + ((lane >> 2) & 1);
}

// 32 entries (TMEM lanes) x 32 columns in tmem_ld_16x32_async's layout -> per column its maximum
// M, the sum S of exp(x - M) and the entry 0..31 of the first maximum (255 without a finite
// logit).  A thread has 4 entries, 8 apart, of each of 8 columns: their state first, then a
// butterfly over the 8 threads that share them, each step folding one half of the columns and
// giving the other away: 21 shuffles and no shared memory (turning 8-column blocks in shared
// memory took 44.2 against 41.4 us at 96 rows, H = 1128, V = 74676).  Entries at or past
// `entries` lie beyond the vocabulary.
__device__ __forceinline__ void wide_reduce_block(const float (&x)[2][16], int entries, int lane,
                                                  float &M, float &S, uint32_t &I)
{
    float m[8], s[8];
    uint32_t id[8];
    const int e0 = lane >> 2;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            v[k] = x[k >> 1][(c >> 1) * 4 + (k & 1) * 2 + (c & 1)];
        if (entries < 32)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                v[k] = e0 + 8 * k < entries ? v[k] : -INFINITY;
        m[c] = fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3]));
        // exp(x - m) as (x - m) * log2e, exact at any magnitude
        const float b = m[c] == -INFINITY ? 0.0f : m[c];
        s[c] = (ex2_mufu((v[0] - b) * kLog2e) + ex2_mufu((v[1] - b) * kLog2e)) +
               (ex2_mufu((v[2] - b) * kLog2e) + ex2_mufu((v[3] - b) * kLog2e));
        const int k = v[0] == m[c] ? 0 : v[1] == m[c] ? 8 : v[2] == m[c] ? 16 : 24;
        id[c] = m[c] == -INFINITY ? 255u : (uint32_t)(e0 + k);
    }
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) {
        const bool hi = (lane & o) != 0;
        const int half = o / 4;
#pragma unroll
        for (int c = 0; c < half; ++c) {
            const float gm = hi ? m[c] : m[c + half], gs = hi ? s[c] : s[c + half];
            const uint32_t gi = hi ? id[c] : id[c + half];
            m[c] = hi ? m[c + half] : m[c];
            s[c] = hi ? s[c + half] : s[c];
            id[c] = hi ? id[c + half] : id[c];
            const float rm = __shfl_xor_sync(0xFFFFFFFFu, gm, o);
            const float rs = __shfl_xor_sync(0xFFFFFFFFu, gs, o);
            const uint32_t ri = __shfl_xor_sync(0xFFFFFFFFu, gi, o);
            wide_fold(m[c], s[c], id[c], rm, rs, ri);
        }
    }
    M = m[0];
    S = s[0];
    I = id[0];
}

// bar.red over the epilogue warps: true when every thread's `ok` is true.
__device__ __forceinline__ bool epilogue_all(bool ok)
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
                 "barrier.cta.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(r)
                 : "r"((uint32_t)ok), "n"(kWideWarps * 32)
                 : "memory");
    return r != 0;
}

template <int EPI>
__global__ void __launch_bounds__(kWideThreads, 1)
    lmhead_wide_kernel(const __grid_constant__ WideRowMaps maps_h,
                       const __grid_constant__ CUtensorMap map_w, const GemmArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t ring_bytes =
        (uint32_t)(kWideSmemBytes - kWideFixed - (size_t)(smem - smem_raw)) / 1024 * 1024;
    uint8_t *fixed = smem + ring_bytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(fixed);
    uint64_t *empty = full + kWideMaxStages;
    uint64_t *tfull = empty + kWideMaxStages;
    uint64_t *tempty = tfull + 4;
    uint64_t *done = tempty + 4;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    float *q_M = reinterpret_cast<float *>(fixed + kWideBarBytes);  // [4][256]
    float *q_S = q_M + 4 * kWideMaxGroup;
    uint8_t *q_I = reinterpret_cast<uint8_t *>(q_S + 4 * kWideMaxGroup);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kWideMaxStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(&tfull[i], 1);
            mbar_init(&tempty[i], 2 * kWideWarps);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        fence_mbar_init();
        tc::prefetch_tensormap(&map_w);
    }
    if (warp == 1)
        tc::tmem_alloc_pair(tmem_slot, kTmemCols);
    tc::fence_before_sync();
    __syncthreads();
    tc::cluster_sync();  // the peer's barriers are initialised before any remote signal
    tc::fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;

    pdl_wait();  // the packed rows and their count are complete

    const int rank = (int)tc::cluster_ctarank();
    const int R = __shfl_sync(0xFFFFFFFFu, *a.row_count, 0);
    const WideCut cut = wide_cut(R);
    const int h = a.wide_h;
    // a CTA's share of a group of g rows in a stage
    auto half_bytes = [](int g) { return (uint32_t)(g / 2 * BK * 2); };
    const uint32_t a_bytes = (uint32_t)(h * BK * 2);
    const uint32_t stage_bytes = a_bytes + half_bytes(cut.g) + half_bytes(cut.g1);
    const int stages = min(kWideMaxStages, (int)(ring_bytes / stage_bytes));
    const WideItems items(cut, a.w_tiles, (int)tc::cluster_count_x(), (int)tc::cluster_id_x());

    // Warps 0 and 1 run whole, one elected lane issuing: loop state and operand addresses then
    // stay warp-uniform, which the issuing instructions need them to be.
    if (warp == 0) {
        const uint64_t pol = make_evict_first_policy();  // W is read once (per row block)
        int s = 0;
        uint32_t ph = 0, filled = 0;
        bool ok = true;
        WidePiece p;
        for (int i = 0; ok && items.piece(i, p); ++i) {
            const bool two = p.w1 != 0;
            const int row0 = p.row0 + rank * (p.w0 / 2);
            const int row1 = p.row0 + p.w0 + rank * (p.w1 / 2);
            const CUtensorMap *map0 = &maps_h.m[p.w0 / 32 - 1];
            const CUtensorMap *map1 = &maps_h.m[two ? p.w1 / 32 - 1 : 0];
            const int w_row = (2 * p.n + rank) * h;
            const uint32_t bytes = a_bytes + half_bytes(p.w0) + half_bytes(p.w1);
            for (int kb = 0; kb < a.k_blocks; ++kb) {
                if (!warp_wait(&empty[s], ph ^ 1u, a.status, abort_flag)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    // Both CTAs' bytes complete on the even CTA's barrier, which it arms.
                    if (rank == 0)
                        mbar_arrive_expect_tx(&full[s], 2 * bytes);
                    const uint32_t bar0 = tc::map_to_rank(&full[s], 0);
                    uint8_t *stage = smem + s * stage_bytes;
                    tc::tma_load_2d_pair_hint(stage, &map_w, kb * BK, w_row, bar0, pol);
                    tc::tma_load_2d_pair(stage + a_bytes, map0, kb * BK, row0, bar0);
                    if (two)
                        tc::tma_load_2d_pair(stage + a_bytes + half_bytes(p.w0), map1, kb * BK,
                                             row1, bar0);
                }
                filled = min(filled + 1, (uint32_t)stages);
                if (++s == stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        // No copy may still be in flight when the pair exits (the odd CTA leaves only after
        // the even one, at the final cluster barrier): the last fill of each stage.
        if (rank == 0 && elect_one())
            drain_ring(full, stages, s, ph, filled, a.status);
        __syncwarp();
    } else if (warp == 1) {
        if (rank == 0) {
            int s = 0;
            uint32_t ph = 0;
            uint32_t used = 0;  // groups accumulated so far
            bool ok = true;
            WidePiece p;
            for (int i = 0; ok && items.piece(i, p); ++i) {
                const bool two = p.w1 != 0;
                const uint32_t b0 = used % cut.buffers, b1 = (used + 1) % cut.buffers;
                const uint32_t turn1 = (used + 1) / cut.buffers;
                if (!warp_wait(&tempty[b0], (used / cut.buffers & 1u) ^ 1u, a.status, abort_flag))
                    break;
                tc::fence_after_sync();
                const uint32_t d0 = tmem_base + b0 * cut.g, d1 = tmem_base + b1 * cut.g;
                const uint32_t idesc0 = tc::idesc_bf16_f32(2 * BM, p.w0);
                const uint32_t idesc1 = tc::idesc_bf16_f32(2 * BM, p.w1);
                // Two groups share each stage.  While the second group's accumulator is still
                // being read, the first one runs ahead over the stages of the ring (k0, at s);
                // the second one follows (k1, at s1), the last to read a stage.
                bool free1 = !two;
                int k0 = 0, k1 = 0, s1 = s;
                while (k1 < a.k_blocks) {
                    if (k0 == k1 || (!free1 && k0 < a.k_blocks && k0 - k1 < stages)) {
                        if (!warp_wait(&full[s], ph, a.status, abort_flag)) {
                            ok = false;
                            break;
                        }
                        tc::fence_after_sync();
                        const uint64_t ad = tc::sw128_kmajor_desc(smem + s * stage_bytes);
                        const uint64_t bd = ad + (a_bytes >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < BK / 16; ++k)
                                tc::mma_bf16_pair(d0, ad + 2u * k, bd + 2u * k, idesc0,
                                                  (k0 | k) != 0);
                            if (!two)
                                tc::commit_pair_multicast(&empty[s]);
                            if (k0 == a.k_blocks - 1)
                                tc::commit_pair_multicast(&tfull[b0]);
                        }
                        ++k0;
                        if (++s == stages) {
                            s = 0;
                            ph ^= 1u;
                        }
                        if (!two) {
                            ++k1;
                            continue;
                        }
                        if (!free1) {
                            free1 = __all_sync(0xFFFFFFFFu,
                                               mbar_try_wait(&tempty[b1], (turn1 & 1u) ^ 1u));
                            if (!free1 && k0 < a.k_blocks && k0 - k1 < stages)
                                continue;
                            if (!free1 && !warp_wait(&tempty[b1], (turn1 & 1u) ^ 1u, a.status,
                                                     abort_flag)) {
                                ok = false;
                                break;
                            }
                            free1 = true;
                            tc::fence_after_sync();
                        }
                    }
                    const uint64_t ad = tc::sw128_kmajor_desc(smem + s1 * stage_bytes);
                    const uint64_t bd = ad + (a_bytes >> 4) + (half_bytes(p.w0) >> 4);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k)
                            tc::mma_bf16_pair(d1, ad + 2u * k, bd + 2u * k, idesc1, (k1 | k) != 0);
                        tc::commit_pair_multicast(&empty[s1]);
                    }
                    ++k1;
                    if (++s1 == stages)
                        s1 = 0;
                }
                if (!ok)
                    break;
                if (two && elect_one())
                    tc::commit_pair_multicast(&tfull[b1]);
                used += two ? 2 : 1;
            }
            // Tensor memory is freed below only after every MMA issued here has completed.
            __syncwarp();
            if (elect_one()) {
                tc::commit_pair_multicast(done);  // the odd CTA's copy is never waited on
                mbar_wait(done, 0, a.status, kDrainLimitNs);
            }
        }
        __syncwarp();
    } else {
        // Epilogue: warp w reads TMEM lanes [32 (w % 4), +32) and every kWideSplit-th block of 32
        // columns.
        const int quarter = warp & 3, third = (warp - 2) >> 2;
        const int et = threadIdx.x - 64;
        uint32_t used = 0;
        bool ok = true;
        WidePiece p;
        for (int i = 0; ok && items.piece(i, p); ++i) {
            const int n = p.n, ng = p.w1 != 0 ? 2 : 1;
            const int ent0 = (2 * n + rank) * h;  // this CTA's entries: ent0 .. ends - 1
            const int ends = min(a.V, ent0 + h);
            for (int j = 0; j < ng; ++j, ++used) {
                const uint32_t buf = used % cut.buffers, turn = used / cut.buffers;
                const bool got = wait_or_abort(&tfull[buf], turn & 1u, a.status, abort_flag);
                // All epilogue warps go on or leave together (they share barriers below); past
                // this one the last group's quarter results have been read.
                if (!epilogue_all(got)) {
                    ok = false;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t taddr =
                    tmem_base + ((uint32_t)(quarter * 32) << 16) + buf * cut.g;
                const int row0 = p.row0 + j * p.w0;
                const int live = min(j == 0 ? p.w0 : p.w1, R - row0);  // columns that are rows
#pragma unroll 1
                for (int c = third * 32; c < live; c += kWideSplit * 32) {
                    float x[2][16];
                    if (EPI == kStore) {  // a lane holds 32 rows' logits of its entry
                        tc::tmem_ld_16cols_async(taddr + c, x[0]);
                        tc::tmem_ld_16cols_async(taddr + c + 16, x[1]);
                    } else {
                        tc::tmem_ld_16x32_async(taddr + c, x[0]);
                        tc::tmem_ld_16x32_async(taddr + (16u << 16) + c, x[1]);
                    }
                    tc::tmem_wait_ld();
                    tc::tie_regs(x[0]);
                    tc::tie_regs(x[1]);
                    if (EPI == kStore) {
                        const int ent = ent0 + quarter * 32 + lane;
                        const int mine = c + lane < live ? a.row_ids[row0 + c + lane] : 0;
#pragma unroll
                        for (int k = 0; k < 32; ++k) {
                            const int64_t row = __shfl_sync(0xFFFFFFFFu, mine, k);
                            if (c + k < live && ent < ends)
                                a.logits[row * a.V + ent] = x[k / 16][k % 16];
                        }
                    } else {
                        float M, S;
                        uint32_t I;
                        wide_reduce_block(x, ends - (ent0 + quarter * 32), lane, M, S, I);
                        const int at = quarter * kWideMaxGroup + c + wide_column(lane);
                        q_M[at] = M;
                        q_S[at] = S;
                        q_I[at] = (uint8_t)I;
                    }
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    if (rank != 0)
                        tc::mbar_arrive_remote(tc::map_to_rank(&tempty[buf], 0));
                    else
                        mbar_arrive(&tempty[buf]);
                }
                if (EPI == kReduce) {
                    asm volatile("barrier.cta.sync 2, %0;" ::"n"(kWideWarps * 32) : "memory");
                    if (et < live) {  // one row's four quarters, in entry order
                        float M = -INFINITY, S = 0.0f;
                        uint32_t I = kNoIdx;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const uint32_t e = q_I[q * kWideMaxGroup + et];
                            fold_state(M, S, I, q_M[q * kWideMaxGroup + et],
                                       q_S[q * kWideMaxGroup + et],
                                       e < 32 ? (uint32_t)(ent0 + q * 32) + e : kNoIdx);
                        }
                        UnitPartial u;
                        u.M = S != S ? __int_as_float(0x7FC00000) : M;
                        u.S = M == -INFINITY ? 0.0f : S;
                        u.idx = I;
                        u.pad = 0;
                        a.partials[(int64_t)(row0 + et) * a.n_tiles + 2 * n + rank] = u;
                    }
                }
            }
        }
    }
    if (threadIdx.x == 0)
        pdl_launch_dependents();  // the row combination may start launching
    __syncthreads();
    tc::cluster_sync();  // both CTAs are done with the pair's tensor memory
    if (warp == 1) {
        __syncwarp();
        tc::fence_after_sync();
        tc::tmem_dealloc_pair(tmem_base, kTmemCols);
    }
    tc::cluster_sync();  // no CTA leaves while its peer may still write into it
}

// Bytes of v that are not zero.
__device__ __forceinline__ int count_nonzero(const uint4 &v)
{
    return __popc(__vsetne4(v.x, 0u)) + __popc(__vsetne4(v.y, 0u)) + __popc(__vsetne4(v.z, 0u)) +
           __popc(__vsetne4(v.w, 0u));
}

// The masked rows packed: their indices (ascending) in row_ids, their number in *row_count and
// their hidden states, in order, in `packed` [row_count][H].  A CTA takes kPackRows neighbouring
// rows, two warps each, and counts the masked rows before them itself (one 16-byte load per
// thread up to 4096 rows), with the rows' own loads in flight meanwhile.  A compaction in one CTA
// and a copy that waited for it took 1.5 us longer (fdllm_lmhead_logits on 192 rows of 50001,
// H = 2048: 45.1 against 43.5 us).
constexpr int kPackRows = 4;
constexpr int kPackThreads = 64 * kPackRows;

__global__ void __launch_bounds__(kPackThreads)
    pack_rows_kernel(const uint8_t *mask, int rows, const int4 *hidden, int64_t vec_per_row,
                     int32_t *row_ids, int32_t *row_count, int4 *packed)
{
    __shared__ int s_cnt[kPackThreads / 32];
    pdl_wait();  // the mask's and the hidden states' writers have completed
    if (threadIdx.x == 0)
        pdl_launch_dependents();  // the GEMM may start its prologue
    const int row0 = blockIdx.x * kPackRows;
    const int mine = threadIdx.x >> 6, t = threadIdx.x & 63;  // this thread's row, place in it
    bool on[kPackRows];
#pragma unroll
    for (int j = 0; j < kPackRows; ++j)
        on[j] = row0 + j < rows && mask[row0 + j] != 0;
    int cnt = 0;
    if ((reinterpret_cast<uintptr_t>(mask) & 15u) == 0) {
        const int whole = row0 / 16;
        for (int i = threadIdx.x; i < whole; i += kPackThreads)
            cnt += count_nonzero(__ldcg(reinterpret_cast<const uint4 *>(mask) + i));
        if (threadIdx.x < row0 - whole * 16)
            cnt += mask[whole * 16 + threadIdx.x] != 0;
    } else {
        for (int i = threadIdx.x; i < row0; i += kPackThreads)
            cnt += mask[i] != 0;
    }
    const bool copies = mine == 0 ? on[0] : mine == 1 ? on[1] : mine == 2 ? on[2] : on[3];
    const int4 *src = hidden + (int64_t)(row0 + mine) * vec_per_row;
    constexpr int kAhead = 8;  // 16-byte loads in flight per thread: a row of H = 4096
    int4 v[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
        if (copies && t + 64 * i < vec_per_row)
            v[i] = __ldg(src + t + 64 * i);
    cnt = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)cnt);
    if ((threadIdx.x & 31) == 0)
        s_cnt[threadIdx.x >> 5] = cnt;
    __syncthreads();
    int k = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kPackThreads / 32; ++w)
        k += s_cnt[w];
    total = k;
#pragma unroll
    for (int j = 0; j < kPackRows; ++j) {
        total += on[j];
        k += j < mine && on[j];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0)
        *row_count = total;
    if (!copies)
        return;
    if (t == 0)
        row_ids[k] = row0 + mine;
    int4 *dst = packed + (int64_t)k * vec_per_row;
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
        if (t + 64 * i < vec_per_row)
            dst[t + 64 * i] = v[i];
    for (int64_t i = t + 64 * kAhead; i < vec_per_row; i += 64)
        dst[i] = __ldg(src + i);
}

// The pair variant's rows are packed by two kernels, this list and a copy by one small CTA per row,
// although that takes 2 us longer: 64 x 32 rows back to back, where the board's power limits this
// variant, take 891 us behind them and 902 behind pack_rows_kernel.  Measured, not explained: the
// GEMM's clusters land on the SMs in another order while 2048 such CTAs come and go, perhaps one
// that shares W tiles better between the two dies (clusters handed out in SM order: 903).
//
// One CTA: the packed list of masked rows (ascending) and its length.
__global__ void __launch_bounds__(1024) compact_rows_kernel(const uint8_t *mask, int rows,
                                                            int32_t *row_ids, int32_t *row_count)
{
    __shared__ int warp_sums[32];
    pdl_wait();  // the mask's writer has completed
    if (threadIdx.x == 0)
        pdl_launch_dependents();
    const int per = (rows + blockDim.x - 1) / blockDim.x;
    const int lo = threadIdx.x * per;
    const int hi = lo + per < rows ? lo + per : rows;
    int cnt = 0;
    for (int i = lo; i < hi; ++i)
        cnt += mask[i] != 0;
    // Block exclusive scan of cnt.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o)
            incl += y;
    }
    if (lane == 31)
        warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        int w = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, w, o);
            if (lane >= o)
                w += y;
        }
        if (lane < nw)
            warp_sums[lane] = w;  // inclusive over warps
    }
    __syncthreads();
    int pos = incl - cnt + (warp > 0 ? warp_sums[warp - 1] : 0);
    for (int i = lo; i < hi; ++i)
        if (mask[i] != 0)
            row_ids[pos++] = i;
    if (threadIdx.x == blockDim.x - 1)
        *row_count = pos;
}

// CTA k copies the hidden state of packed row k (16-byte vectors).
__global__ void gather_rows_kernel(const int4 *hidden, int64_t vec_per_row, const int32_t *row_ids,
                                   const int32_t *row_count, int4 *packed)
{
    pdl_wait();  // the row list is complete
    if (threadIdx.x == 0)
        pdl_launch_dependents();  // the GEMM may start its prologue
    const int k = blockIdx.x;
    if (k >= *row_count)
        return;
    const int4 *src = hidden + (int64_t)row_ids[k] * vec_per_row;
    int4 *dst = packed + (int64_t)k * vec_per_row;
    for (int64_t i = threadIdx.x; i < vec_per_row; i += blockDim.x)
        dst[i] = __ldg(src + i);
}

struct Part {
    float M, S;
    uint32_t idx;
    bool nan;
};

// Fold of two partials: larger max, sums re-based to it, the lowest index attaining it.
// Symmetric, so both lanes of a shuffle step obtain the same bits.
__device__ __forceinline__ Part fold(const Part &x, const Part &y)
{
    Part r;
    r.nan = x.nan || y.nan;
    r.M = fmaxf(x.M, y.M);
    r.S = rebase(x.S, x.M, r.M) + rebase(y.S, y.M, r.M);
    const uint32_t ix = x.M == r.M ? x.idx : kNoIdx;
    const uint32_t iy = y.M == r.M ? y.idx : kNoIdx;
    r.idx = ix < iy ? ix : iy;
    return r;
}

__device__ __forceinline__ Part as_part(const int4 &v)
{
    Part y{__int_as_float(v.x), __int_as_float(v.y), (uint32_t)v.z, false};
    y.nan = y.M != y.M;
    if (y.nan)
        y.M = -__int_as_float(0x7F800000);
    return y;
}

__device__ __forceinline__ Part shfl_part(const Part &x, int o)
{
    Part y;
    y.M = __shfl_xor_sync(0xFFFFFFFFu, x.M, o);
    y.S = __shfl_xor_sync(0xFFFFFFFFu, x.S, o);
    y.idx = __shfl_xor_sync(0xFFFFFFFFu, x.idx, o);
    y.nan = __shfl_xor_sync(0xFFFFFFFFu, (int)x.nan, o) != 0;
    return y;
}

// c = min(1/S, 1) and x_hat of a whole row; NaN and -1 with a NaN logit or an infinite maximum.
__device__ __forceinline__ void store_conf(const Part &x, int row, float *conf, int32_t *tok)
{
    const bool finite = fabsf(x.M) <= 3.402823466e38f && fabsf(x.S) <= 3.402823466e38f;
    const bool bad = x.nan || !finite || !(x.S > 0.0f) || x.idx == kNoIdx;
    conf[row] = bad ? __int_as_float(0x7FC00000) : fminf(1.0f / x.S, 1.0f);
    tok[row] = bad ? -1 : (int32_t)x.idx;
}

// One CTA of kCombineWarps warps per packed row: lane l of warp q folds tiles
// q * 32 + l + 128 i (i = 0, 1, ...) in order, the lanes of each warp fold in a fixed
// butterfly, and the warps' results fold in warp order.  A fixed tree, so the result does not
// depend on timing.  Writes c = min(1/S, 1) and x_hat at the row's (b, l); a row with a NaN
// logit or an infinite maximum gets c = NaN, x_hat = -1.
constexpr int kCombineWarps = 4;

__global__ void __launch_bounds__(kCombineWarps * 32)
    combine_rows_kernel(const UnitPartial *partials, int n_tiles, const int32_t *row_ids,
                        const int32_t *row_count, float *conf, int32_t *tok)
{
    __shared__ Part s_part[kCombineWarps];
    pdl_wait();  // every tile partial is written
    if (threadIdx.x == 0)
        pdl_launch_dependents();
    const int r = blockIdx.x;
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    if (r >= *row_count)
        return;
    Part acc{-__int_as_float(0x7F800000), 0.0f, kNoIdx, false};
    const UnitPartial *p = partials + (int64_t)r * n_tiles;
    constexpr int kStride = kCombineWarps * 32;
    constexpr int kBatch = 8;  // loads in flight per lane before the folds
    for (int j0 = q * 32 + lane; j0 < n_tiles; j0 += kStride * kBatch) {
        int4 v[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
            if (j0 + kStride * b < n_tiles)
                v[b] = __ldcg(reinterpret_cast<const int4 *>(p + j0 + kStride * b));
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
            if (j0 + kStride * b < n_tiles)
                acc = fold(acc, as_part(v[b]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        acc = fold(acc, shfl_part(acc, o));
    if (lane == 0)
        s_part[q] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        acc = s_part[0];
        for (int w = 1; w < kCombineWarps; ++w)
            acc = fold(acc, s_part[w]);
        store_conf(acc, row_ids[r], conf, tok);
    }
}

// ----------------------------------------------------------------------------- host side
// Workspace layout (offsets from the 256-byte aligned base; header shared with
// fdllm_select's layout: status at 0, the vocab reduction's counter at 4 left untouched):
//   row_count int32 at 8
//   row_ids   int32 [rows]
//   packed    bf16 [rows][H]            (1024-byte aligned: a TMA source)
//   partials  UnitPartial [rows][n_tiles]
//   conf      fp32 [rows], tok int32 [rows]
struct LmLayout {
    size_t row_count, row_ids, packed, partials, conf, tok, total;
};

size_t up(size_t x, size_t a) { return (x + a - 1) / a * a; }

LmLayout lm_layout(int64_t rows, int64_t H, int64_t n_tiles)
{
    LmLayout l;
    l.row_count = 8;
    l.row_ids = 256;
    l.packed = up(l.row_ids + (size_t)rows * 4, 1024);
    l.partials = up(l.packed + (size_t)rows * H * 2, 256);
    l.conf = up(l.partials + (size_t)rows * n_tiles * sizeof(UnitPartial), 256);
    l.tok = up(l.conf + (size_t)rows * 4, 256);
    l.total = up(l.tok + (size_t)rows * 4, 256);
    return l;
}

using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                   const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                   const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return (EncodeTiledFn) nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// bf16 matrix [outer][inner] (row stride inner * 2 bytes), loaded as boxes of
// {BK, box_outer} with 128-byte swizzling; out-of-range elements read as zero.
bool make_map(CUtensorMap *map, const void *base, int64_t inner, int64_t outer, int box_outer)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc)
        return false;
    const cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
    const cuuint64_t strides[1] = {(cuuint64_t)inner * 2};
    const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_outer};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides,
               box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// A launch as a programmatic dependent of the previous kernel on the stream (in plain
// stream order when pdl is false).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(bool pdl, void (*kern)(KArgs...), unsigned grid, unsigned block,
                       cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

fdllm_status check_lmhead(const void *hidden, const void *w, int B, int L, int H, int V,
                          const uint8_t *mask)
{
    if (B < 1 || L < 1 || L > FDLLM_MAX_L || (int64_t)B * L > FDLLM_MAX_ROWS || V < 1 || H < 8)
        return FDLLM_ERR_ARG;
    if (!hidden || !w || !mask)
        return FDLLM_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(hidden) & 15u) || (reinterpret_cast<uintptr_t>(w) & 15u) ||
        H % 8 != 0)
        return FDLLM_ERR_ALIGN;
    const int64_t n_tiles = (V + 207) / 208;  // the narrowest tile
    if ((int64_t)B * L * n_tiles >= ((int64_t)1 << 31) || (int64_t)H * 2 >= ((int64_t)1 << 31))
        return FDLLM_ERR_ARG;
    return FDLLM_OK;
}

int sm_count();

// The slab variant's tile height: the multiple of 8 in [96, 128] that minimises the W rows
// of the busiest CTA, ceil(ceil(V / h) / P) * h with P = min(tiles, SMs); ties go to the
// taller tile (fewer, larger copies).  Heights below 96 would put too few W bytes in each
// stage to keep the stream going.
int slab_height(int V)
{
    const int64_t sms = sm_count();
    int best = 128;
    int64_t best_rows = -1;
    for (int h = 128; h >= 96; h -= 8) {
        const int64_t tiles = ((int64_t)V + h - 1) / h;
        const int64_t P = tiles < sms ? tiles : sms;
        const int64_t rows = (tiles + P - 1) / P * h;
        if (best_rows < 0 || rows < best_rows) {
            best = h;
            best_rows = rows;
        }
    }
    return best;
}

// The wide variant's W rows per CTA and tile.  A few rows leave it bound by W alone, and the slab
// variant's heights (104 for LLaDA's V: eight whole rounds instead of six and a half) balance
// that: of 128 rows 8 masked 155 against 163 us, 32 157 against 163, 96 158 against 159, 128 160
// against 160.  More rows make it the tensor cores', whose M = 256 a lower tile leaves partly
// unused: of 192 rows all masked 167 against 164, of 256 196 against 178, 288 of 384 225 against
// 195.  So the line lies at 192, by the shape alone: a row's partials must not depend on how many
// rows are masked, and so beyond it a few masked rows take the tall tiles, too (of 256 rows 16
// masked 156 low, 162 tall, 64 157 and 160; with row tiles 158 against 157 tall on another box).
// Measured on LLaDA's V; at V = 50000, H = 4096 256 of 256 rows are level (79 low, 81 tall).
constexpr int kWideLowRows = 192;

int wide_height(int64_t rows, int V)
{
    return rows <= kWideLowRows ? slab_height(V) : BM;
}

// The slab variant's grid: one CTA per SM, or one per tile if there are fewer.
int slab_grid(int V)
{
    const int64_t h = slab_height(V);
    const int64_t tiles = ((int64_t)V + h - 1) / h;
    return (int)(tiles < sm_count() ? tiles : sm_count());
}

// The GEMM variant: the slab variant for at most kSlabRows rows (its row operand is 4 KB per K-block
// where a row tile's is 16 KB, and its busiest CTA never streams more W rows than with row tiles,
// since half of either tile width is one of its heights), then the wide one up to a number of rows,
// the pair beyond.  The pair computes whole tiles of 256 rows, and
// with a short K loop (H up to 2048) its four epilogue warps set its pace: there the wide variant
// stays ahead up to all the rows measured.  With a longer one it is level with the pair at the rows
// of a whole tile and ahead in between and with few rows masked, until the power limit decides
// (passes back to back), where the pair needs 1 to 3 % less.  fdllm_lmhead_confidence, wide / pair,
// us (back to back in brackets):
// H = 4096, V = 126464: of 32 x 32 rows 51 masked 160 / 182, 640 368 / 398, 768 431 / 426 (494 /
// 484); of 40 x 32 640 383 / 413, 800 470 / 507, 1280 684 / 683 (775 / 775); of 48 x 32 76 159 /
// 188, 768 428 / 425, 1100 599 / 642, 1536 808 / 797 (920 / 902); of 64 x 32 102 161 / 189, 1300
// 695 / 740, 1536 813 / 793 (928 / 900), 2048 1070 / 1043; of 96 x 32 3072 1611 / 1535.
// H = 3072, V = 80000: of 1536 1152 334 / 335 (380 / 377); of 2048 102 90 / 106, 2048 512 / 514.
// H = 2560, V = 126464: of 2048 102 106 / 125, 1024 353 / 352, 2048 675 / 671 (767 / 762); of 4096
// 204 114 / 130, 2048 683 / 675, 4096 1346 / 1297 (1508 / 1476).
// H = 2048, V = 126464: of 2048 1536 418 / 429 (479 / 486); of 4096 4096 1084 / 1091 (1217 / 1235).
// H = 1024, V = 100000: of 2048 1536 194 / 319, of 4096 4096 491 / 821.  H = 512, V = 30000: 2048
// 72 / 128.
// fdllm_lmhead_logits, which takes the same variant, H = 4096, V = 50000: 576 of 768 149 / 184, 768
// of 1024 188 / 189, 1152 of 1536 291 / 286 (336 / 325); H = 1024, V = 30000, 1152 of 1536 62 / 108.
// FDLLM_LMHEAD_GEMM = solo, pair, slab or wide forces one (slab only where B * L <= kSlabRows).
constexpr int kWideDeepH = 2560;
constexpr int kWideRowsMax = 4096;          // H <= kWideDeepH: the most rows measured
constexpr int kWideRowsDeep = 48 * 32;      // H beyond

int gemm_mode(int64_t rows, int H, int V)
{
    if (const char *e = std::getenv("FDLLM_LMHEAD_GEMM")) {
        const std::string v(e);
        if (v == "solo")
            return kSolo;
        if (v == "pair")
            return kPair;
        if (v == "slab" && rows <= kSlabRows)
            return kSlab;
        if (v == "wide")
            return kWide;
    }
    if (rows <= kSlabRows)
        return kSlab;
    return rows <= (H <= kWideDeepH ? kWideRowsMax : kWideRowsDeep) ? kWide : kPair;
}

int sm_count()
{
    static std::once_flag once[64];
    static int cache[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return 152;
    std::call_once(once[dev], [&] {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        cache[dev] = n > 0 ? n : 152;
    });
    return cache[dev];
}

// The vocabulary tile width with the least estimated time: whole waves of tiles over the
// SMs (row tiles estimated from B * L, the most the mask can hold) times the tile width.
// Ties go to 208 for one CTA per tile (measured 1.3-1.4 % faster at 4 estimated row tiles,
// B = 14 and 16 of 32 positions) and to 256 for the CTA pair (208 is slower there at every
// size).  FDLLM_LMHEAD_BN = 256 or 208 forces one.
int choose_bn(int64_t rows, int V, bool pair)
{
    if (const char *e = std::getenv("FDLLM_LMHEAD_BN")) {
        const int f = std::atoi(e);
        if (f == 256 || f == 208)
            return f;
    }
    const int64_t m_tiles = (rows + BM - 1) / BM, sms = sm_count();
    const int order[2] = {pair ? 256 : 208, pair ? 208 : 256};  // the first wins ties
    int best = order[0];
    int64_t best_cost = -1;
    for (int bn : order) {
        const int64_t tiles = (V + bn - 1) / bn * m_tiles;
        const int64_t cost = (tiles + sms - 1) / sms * bn;
        if (best_cost < 0 || cost < best_cost) {
            best = bn;
            best_cost = cost;
        }
    }
    return best;
}

template <int EPI, int MODE, int BN>
cudaError_t launch_gemm_cfg(const CUtensorMap &mh, const CUtensorMap &mw, const GemmArgs &g,
                            cudaStream_t stream)
{
    constexpr int CL = MODE == kSolo ? 1 : 2;
    static std::once_flag once[64];
    static int grid[64];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess)
        return err;
    if (dev < 0 || dev >= 64)
        return cudaErrorInvalidDevice;
    auto kern = lmhead_gemm_kernel<EPI, MODE, BN>;
    constexpr size_t smem = TileCfg<BN, MODE, EPI>::kSmemBytes;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;  // the occupancy query below sees the cluster shape only
    std::call_once(once[dev], [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        const int sms = sm_count();
        int clusters = 0;
        cfg.gridDim = dim3((unsigned)(sms / CL * CL));
        if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess || clusters < 1)
            clusters = sms / CL;
        (void)cudaGetLastError();
        grid[dev] = clusters * CL;  // persistent: every cluster resident at once
    });
    cfg.gridDim = dim3((unsigned)grid[dev]);
    cfg.numAttrs = g.pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, mh, mw, g);
}

template <int EPI, int MODE>
cudaError_t launch_gemm_mode(const CUtensorMap &mh, const CUtensorMap &mw, const GemmArgs &g,
                             int bn, cudaStream_t stream)
{
    return bn == 208 ? launch_gemm_cfg<EPI, MODE, 208>(mh, mw, g, stream)
                     : launch_gemm_cfg<EPI, MODE, 256>(mh, mw, g, stream);
}

template <int EPI>
cudaError_t launch_slab(const CUtensorMap &mh, const CUtensorMap &mw, const GemmArgs &g,
                        cudaStream_t stream)
{
    static std::once_flag once[64];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess)
        return err;
    if (dev < 0 || dev >= 64)
        return cudaErrorInvalidDevice;
    auto kern = lmhead_slab_kernel<EPI>;
    std::call_once(once[dev], [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSlabSmemBytes);
    });
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g.n_tiles);
    cfg.blockDim = dim3(kSlabThreads);
    cfg.dynamicSmemBytes = kSlabSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, mh, mw, g);
}

template <int EPI>
cudaError_t launch_wide(const WideRowMaps &mh, const CUtensorMap &mw, const GemmArgs &g,
                        cudaStream_t stream)
{
    static std::once_flag once[64];
    static int grid[64];
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess)
        return err;
    if (dev < 0 || dev >= 64)
        return cudaErrorInvalidDevice;
    auto kern = lmhead_wide_kernel<EPI>;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kWideThreads);
    cfg.dynamicSmemBytes = kWideSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;  // the occupancy query below sees the cluster shape only
    std::call_once(once[dev], [&] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kWideSmemBytes);
        const int sms = sm_count();
        int clusters = 0;
        cfg.gridDim = dim3((unsigned)(sms / 2 * 2));
        if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess || clusters < 1)
            clusters = sms / 2;
        (void)cudaGetLastError();
        grid[dev] = clusters * 2;  // persistent: every pair resident at once
    });
    cfg.gridDim = dim3((unsigned)grid[dev]);
    cfg.numAttrs = g.pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, mh, mw, g);
}

template <int EPI>
cudaError_t launch_gemm(const CUtensorMap &mh, const CUtensorMap &mw, const GemmArgs &g,
                        int mode, int bn, cudaStream_t stream)
{
    if (mode == kSlab)
        return launch_slab<EPI>(mh, mw, g, stream);
    switch (mode) {
    case kPair: return launch_gemm_mode<EPI, kPair>(mh, mw, g, bn, stream);
    default: return launch_gemm_mode<EPI, kSolo>(mh, mw, g, bn, stream);
    }
}

// How one call is cut, and its workspace.
struct LmPlan {
    int mode, bn;  // bn: W rows of a tile (per CTA in the wide variant)
    int w_tiles;   // tiles of 2 bn W rows
    int n_tiles;   // partials per row: one per vocabulary tile (per CTA of the pair in the wide
                   // variant), or one per CTA of the slab variant
    LmLayout lay;
};

LmPlan lm_plan(int mode, int64_t rows, int H, int V)
{
    LmPlan p;
    p.mode = mode;
    p.bn = mode == kSlab   ? slab_height(V)
           : mode == kWide ? wide_height(rows, V)
                           : choose_bn(rows, V, mode == kPair);
    p.w_tiles = (V + 2 * p.bn - 1) / (2 * p.bn);
    p.n_tiles = mode == kSlab   ? slab_grid(V)
                : mode == kWide ? 2 * p.w_tiles
                                : (V + p.bn - 1) / p.bn;
    p.lay = lm_layout(rows, H, p.n_tiles);
    return p;
}

// Steps 1-2 (and 3 for the reduce epilogue) on the owned workspace.  The confidences and
// argmaxes go to conf and tok [B, L], or to the workspace where those are null.
fdllm_status run_lmhead(const void *hidden, const void *w, int B, int L, int H, int V,
                        const uint8_t *mask, int epi, float *out_logits, cudaStream_t s,
                        uint8_t **ws_out, LmLayout *lay_out, bool pdl = true,
                        float *conf = nullptr, int32_t *tok = nullptr)
{
    const int64_t rows = (int64_t)B * L;
    LmPlan plan = lm_plan(gemm_mode(rows, H, V), rows, H, V);
    // The workspace does not grow under capture; one that calls of other shapes have sized may hold
    // only the tile variants' partials, which are fewer.
    if (plan.mode == kWide && !owned_workspace_ready(plan.lay.total, s))
        plan = lm_plan((rows + BM - 1) / BM >= 8 ? kPair : kSolo, rows, H, V);
    const int mode = plan.mode, bn = plan.bn, n_tiles = plan.n_tiles;
    const LmLayout lay = plan.lay;
    void *wsv = nullptr;
    fdllm_status st = owned_workspace(lay.total, lmhead_reserve_bytes(rows, H, V), s, &wsv);
    if (st != FDLLM_OK)
        return st;
    uint8_t *ws = static_cast<uint8_t *>(wsv);
    int32_t *row_count = reinterpret_cast<int32_t *>(ws + lay.row_count);
    int32_t *row_ids = reinterpret_cast<int32_t *>(ws + lay.row_ids);
    uint8_t *packed = ws + lay.packed;

    CUtensorMap mh, mw;
    WideRowMaps wide_maps;
    if (!make_map(&mw, w, H, V, mode == kPair ? bn / 2 : bn))
        return FDLLM_ERR_CUDA;
    if (mode == kWide) {
        for (int i = 0; i < kWideMaps && 32 * i < rows; ++i)  // groups no wider than the rows
            if (!make_map(&wide_maps.m[i], packed, H, rows, 16 * (i + 1)))
                return FDLLM_ERR_CUDA;
    } else if (!make_map(&mh, packed, H, rows, mode == kSlab ? kSlabRows : BM)) {
        return FDLLM_ERR_CUDA;
    }

    if (mode == kPair) {
        if (launch_pdl(pdl, compact_rows_kernel, 1, 1024, s, mask, (int)rows, row_ids,
                       row_count) != cudaSuccess ||
            launch_pdl(pdl, gather_rows_kernel, (unsigned)rows, 128, s,
                       static_cast<const int4 *>(hidden), (int64_t)(H / 8),
                       (const int32_t *)row_ids, (const int32_t *)row_count,
                       reinterpret_cast<int4 *>(packed)) != cudaSuccess)
            return FDLLM_ERR_CUDA;
    } else if (launch_pdl(pdl, pack_rows_kernel, (unsigned)((rows + kPackRows - 1) / kPackRows),
                          kPackThreads, s, mask, (int)rows, static_cast<const int4 *>(hidden),
                          (int64_t)(H / 8), row_ids, row_count,
                          reinterpret_cast<int4 *>(packed)) != cudaSuccess) {
        return FDLLM_ERR_CUDA;
    }
    GemmArgs g;
    g.row_count = row_count;
    g.row_ids = row_ids;
    g.V = V;
    g.n_tiles = n_tiles;
    g.k_blocks = (H + BK - 1) / BK;
    g.slab_h = mode == kSlab ? bn : 0;
    g.slab_tiles = mode == kSlab ? (V + bn - 1) / bn : 0;
    g.w_tiles = plan.w_tiles;
    g.wide_h = mode == kWide ? bn : 0;
    g.partials = reinterpret_cast<UnitPartial *>(ws + lay.partials);
    g.logits = out_logits;
    g.status = reinterpret_cast<uint32_t *>(ws);
    g.pdl = pdl;
    cudaError_t e;
    if (mode == kWide)
        e = epi == kReduce ? launch_wide<kReduce>(wide_maps, mw, g, s)
                           : launch_wide<kStore>(wide_maps, mw, g, s);
    else
        e = epi == kReduce ? launch_gemm<kReduce>(mh, mw, g, mode, bn, s)
                           : launch_gemm<kStore>(mh, mw, g, mode, bn, s);
    if (e != cudaSuccess)
        return FDLLM_ERR_CUDA;
    if (!conf)
        conf = reinterpret_cast<float *>(ws + lay.conf);
    if (!tok)
        tok = reinterpret_cast<int32_t *>(ws + lay.tok);
    if (epi == kReduce) {
        if (launch_pdl(pdl, combine_rows_kernel, (unsigned)rows, kCombineWarps * 32, s,
                       (const UnitPartial *)g.partials, n_tiles, (const int32_t *)row_ids,
                       (const int32_t *)row_count, conf, tok) != cudaSuccess)
            return FDLLM_ERR_CUDA;
    }
    *ws_out = ws;
    *lay_out = lay;
    return FDLLM_OK;
}

}  // namespace
}  // namespace fdllm

using namespace fdllm;

namespace fdllm {

size_t lmhead_need_bytes(int64_t rows, int H, int V)
{
    return lm_plan(gemm_mode(rows, H, V), rows, H, V).lay.total;
}

// The wide variant keeps up to twice the pair's partials per row, lower tiles more again, and how
// far up it serves depends on H: the need of a call falls in places as its shape grows.
size_t lmhead_reserve_bytes(int64_t rows, int H, int V)
{
    auto bytes = [](int64_t r, int h, int64_t n_tiles) { return lm_layout(r, h, n_tiles).total; };
    const int64_t wide = 2 * (((int64_t)V + 255) / 256);
    return std::max({bytes(rows, H, ((int64_t)V + 207) / 208),
                     bytes(std::min<int64_t>(rows, kWideLowRows), H, 2 * (((int64_t)V + 191) / 192)),
                     bytes(std::min<int64_t>(rows, kWideRowsDeep), H, wide),
                     bytes(std::min<int64_t>(rows, kWideRowsMax), std::min(H, kWideDeepH), wide)});
}

fdllm_status lmhead_select_owned(const void *hidden, const void *w_vocab, int B, int L, int H,
                                 int V, uint8_t *mask, double param, int mode,
                                 int32_t *out_tokens, uint8_t *out_commit, int32_t *out_n,
                                 cudaStream_t s, bool pdl)
{
    fdllm_status st = check_lmhead(hidden, w_vocab, B, L, H, V, mask);
    if (st != FDLLM_OK)
        return st;
    if (!out_tokens || !out_commit || !out_n || !std::isfinite(param) ||
        (mode != FDLLM_PROFILE && mode != FDLLM_FACTOR && mode != FDLLM_THRESHOLD))
        return FDLLM_ERR_ARG;
    uint8_t *ws = nullptr;
    LmLayout lay;
    st = run_lmhead(hidden, w_vocab, B, L, H, V, mask, kReduce, nullptr, s, &ws, &lay, pdl);
    if (st != FDLLM_OK)
        return st;
    ProfileSelectArgs pa;
    pa.units_per_row = 0;
    pa.partials = nullptr;
    pa.next_unit = nullptr;
    pa.conf = reinterpret_cast<const float *>(ws + lay.conf);
    pa.tok = reinterpret_cast<const int32_t *>(ws + lay.tok);
    pa.mask = mask;
    pa.B = B;
    pa.L = L;
    pa.mode = mode;
    pa.param = param;
    pa.eta = 0.0;
    pa.eta_pos = nullptr;
    pa.out_tokens = out_tokens;
    pa.out_commit = out_commit;
    pa.out_n = out_n;
    pa.status = reinterpret_cast<uint32_t *>(ws);
    pa.pdl = pdl;
    return launch_profile_select(pa, s) == cudaSuccess ? FDLLM_OK : FDLLM_ERR_CUDA;
}

}  // namespace fdllm

extern "C" {

fdllm_status fdllm_lmhead_select(const void *hidden, const void *w_vocab, int B, int L, int H,
                                 int V, uint8_t *mask, double param, int mode,
                                 int32_t *out_tokens, uint8_t *out_commit, int32_t *out_n,
                                 void *stream)
{
    return lmhead_select_owned(hidden, w_vocab, B, L, H, V, mask, param, mode, out_tokens,
                               out_commit, out_n, static_cast<cudaStream_t>(stream), true);
}

fdllm_status fdllm_lmhead_confidence(const void *hidden, const void *w_vocab, int B, int L,
                                     int H, int V, const uint8_t *mask, float *out_conf,
                                     int32_t *out_argmax, void *stream)
{
    fdllm_status st = check_lmhead(hidden, w_vocab, B, L, H, V, mask);
    if (st != FDLLM_OK)
        return st;
    if (!out_conf || !out_argmax)
        return FDLLM_ERR_ARG;
    uint8_t *ws = nullptr;
    LmLayout lay;
    return run_lmhead(hidden, w_vocab, B, L, H, V, mask, kReduce, nullptr,
                      static_cast<cudaStream_t>(stream), &ws, &lay, true, out_conf, out_argmax);
}

fdllm_status fdllm_lmhead_logits(const void *hidden, const void *w_vocab, int B, int L, int H,
                                 int V, const uint8_t *mask, float *out_logits, void *stream)
{
    fdllm_status st = check_lmhead(hidden, w_vocab, B, L, H, V, mask);
    if (st != FDLLM_OK)
        return st;
    if (!out_logits)
        return FDLLM_ERR_ARG;
    uint8_t *ws = nullptr;
    LmLayout lay;
    return run_lmhead(hidden, w_vocab, B, L, H, V, mask, kStore, out_logits,
                      static_cast<cudaStream_t>(stream), &ws, &lay);
}

}  // extern "C"
