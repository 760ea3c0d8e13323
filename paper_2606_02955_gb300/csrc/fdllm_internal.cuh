// fdllm_internal.cuh -- what the kernels and the C interface share: argument blocks,
// workspace pieces, launch entry points and the per-row combination of unit results.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "fdllm.h"

namespace fdllm {

// ------------------------------------------------------------------ vocab reduction (a1)
// Each row of logits is cut into units_per_row units of unit_vecs 16-byte vectors (the last
// unit may be shorter), with units_per_row = ceil(row_bytes / target).  A unit is reduced by
// one CTA in a fixed order, so a row's result depends only on its bytes and the call's
// shape (B * L, V, dtype), which fixes the plan.  The CTA streams a unit through a ring of
// shared-memory chunk buffers.  The target is 128 KB; a step whose logits, all B * L rows
// counted, fit in about one wave of such units over the SMs (kSmallStepBytes) takes 64 KB
// units instead, so that twice as many SMs share its reduction: there the per-SM exp
// throughput and the first copy's latency, not HBM, set the time.  A smaller unit does not
// fill the ring (192 KB in flight per SM), so short rows take warp units (below).
constexpr int kSegQueue = 8;  // unit results queued from math warps to the epilogue warp
constexpr int64_t kUnitTargetBytes = 131072;
constexpr int64_t kSmallUnitTargetBytes = 65536;
constexpr int64_t kSmallStepBytes = 20ll << 20;
constexpr int kMaxGrid = 1024;
constexpr int kMaxRows = 65536;
constexpr int kMaskWords = kMaxRows / 32;

constexpr float kLog2e = 1.4426950408889634f;
constexpr uint32_t kNoIdx = 0xFFFFFFFFu;

// Reduction of one unit (or one vocabulary tile or slab of the LM head): max logit M,
// S = sum of exp(x - M) over it, relative to M exactly (see rebase_scaled), and the
// row-relative index of the first logit equal to M.
struct UnitPartial {
    float M;
    float S;
    uint32_t idx;
    uint32_t pad;
};

struct VocabReduceArgs {
    const uint8_t *logits;   // [rows, V] element size esize
    const uint8_t *mask;     // [rows]
    int64_t rows;            // B * L
    int64_t row_bytes;       // V * esize
    int64_t vec_per_row;     // row_bytes / 16
    int32_t units_per_row;
    int32_t unit_vecs;
    UnitPartial *partials;   // [rows][units_per_row]; written for masked rows
    uint32_t *next_unit;     // work queue past the first gridDim.x units: zero on entry,
                             // zero again after the launch's last fetch
    uint32_t *status;        // sticky device error bits
    bool pdl = true;         // launch as a programmatic dependent of the previous kernel
    bool warp_units = false; // the units are warp units (UnitPlan)
};

struct UnitPlan {
    int32_t units_per_row;
    int32_t unit_vecs;
    bool warp_units;  // one warp reduces a unit, otherwise one CTA
};

// Unit lengths are rounded up to a multiple of kUnitAlignVecs vectors (8 KB), so that every
// unit but a row's last one fills whole chunks; the unit count is then recomputed so that
// no unit is empty.
constexpr int64_t kUnitAlignVecs = 512;

// Short rows.  A unit reduced by a whole CTA pays a ring hand-over and a 16-warp reduction
// (about 1.4 us) and has only itself in flight, so where a row is one unit of at most 64 KB
// the units are warp units instead: one warp each, 32 in flight per SM.  Measured per launch,
// CTA units against warp units: 1004 fp32 logits x 44100 rows 403 against 34 us, 4096 bf16 x
// 6554 rows 66 against 14, 20008 fp16 x 6393 rows 67 against 42, 32000 bf16 x 1434 rows 19.1
// against 19.0 (level: the bound on the row), 50304 bf16 x 1434 rows 28.9 against 29.0, and
// 50304 fp32 x 1434 rows 43.9 against 47.0.  With at most two rows per SM a CTA spreads a
// row over more lanes: 20008 bf16 x 32 rows 4.1 against 5.6 us, x 205 rows 6.6 against 6.4.
// 8 KB units measured fastest (128, 256, 512 and 1024 vectors: 50.2, 50.2, 42.2 and 44.3 us at
// 20008 fp16), and at most 8 of them let one thread fold a position's partials in one round.
constexpr int64_t kWarpRowBytes = 65536;
constexpr int64_t kWarpMinRows = 2 * 152;
constexpr int64_t kWarpUnitVecs = 512;
static_assert(kWarpRowBytes / 16 / kWarpUnitVecs <= 8, "partials folded in one round");
// Beyond one per row, no more warp units than the static scratch array has room for.
constexpr int64_t kMostWarpUnits =
    (FDLLM_STATIC_SCRATCH_BYTES - 256) / (int64_t)sizeof(UnitPartial);

// warp_units = false plans CTA units whatever the shape: one partial per short row, for scratch
// memory that does not hold more (see layout_within).
inline UnitPlan plan_units(int64_t row_bytes, int64_t rows, bool warp_units = true)
{
    const int64_t vpr = row_bytes / 16;
    if (warp_units && row_bytes <= kWarpRowBytes && rows > kWarpMinRows) {
        const int64_t fit = kMostWarpUnits / rows;
        int64_t upr = (vpr + kWarpUnitVecs - 1) / kWarpUnitVecs;
        upr = upr > fit ? fit : upr;
        upr = upr < 1 ? 1 : upr;
        const int64_t uv = ((vpr + upr - 1) / upr + 31) / 32 * 32;
        return UnitPlan{(int32_t)((vpr + uv - 1) / uv), (int32_t)uv, true};
    }
    const int64_t target =
        rows * row_bytes <= kSmallStepBytes ? kSmallUnitTargetBytes : kUnitTargetBytes;
    int64_t upr = (row_bytes + target - 1) / target;
    if (upr < 1)
        upr = 1;
    int64_t uv = (vpr + upr - 1) / upr;
    uv = (uv + kUnitAlignVecs - 1) / kUnitAlignVecs * kUnitAlignVecs;
    upr = (vpr + uv - 1) / uv;
    if (upr < 1)
        upr = 1;
    return UnitPlan{(int32_t)upr, (int32_t)uv, false};
}

// Enqueue the vocab reduction on all SMs, as a programmatic dependent of the previous
// kernel on the stream.
cudaError_t launch_vocab_reduce(const VocabReduceArgs &a, int dtype, cudaStream_t stream);

// One thread waits, bounded by limit_ns, on an mbarrier that never completes.
cudaError_t launch_bounded_wait_probe(uint32_t *status, uint64_t limit_ns, cudaStream_t stream);

// Per masked position: combine its unit partials, write (c, x_hat); resets next_unit.
// Launched as a programmatic dependent of the vocab reduction.
struct FinalizeArgs {
    const uint8_t *mask;
    int64_t rows;
    int32_t units_per_row;
    const UnitPartial *partials;
    float *out_conf;
    int32_t *out_tok;
    uint32_t *next_unit;
    bool warp_units;  // the partials come from warp units
};

cudaError_t launch_finalize(const FinalizeArgs &a, cudaStream_t stream);

// ------------------------------------------------------------------ profile select (a2-a5)
// The profile rule on calibration-robust lower confidences max{0, c - eta} (App. C).
constexpr int kModeRobust = 3;

struct ProfileSelectArgs {
    // Source of (c, x_hat): unit partials (from the vocab reduction, which this kernel then
    // follows as a programmatic dependent launch) when `partials` is non-null, otherwise the
    // given conf/tok arrays.
    int32_t units_per_row;
    const UnitPartial *partials;
    uint32_t *next_unit;     // reset to zero when partials are consumed
    const float *conf;       // [B, L]
    const int32_t *tok;      // [B, L]
    uint8_t *mask;           // [B, L], updated in place
    int B;
    int L;
    int mode;                // 0 profile, 1 factor, 2 threshold, kModeRobust
    double param;
    double eta;              // kModeRobust: uniform calibration allowance
    const float *eta_pos;    // kModeRobust: [B, L] per-position allowances, or null
    int32_t *out_tokens;     // [B, L]
    uint8_t *out_commit;     // [B, L]
    int32_t *out_n;          // [B]
    uint32_t *status;        // nullable: the timeout bit set -> every row reports a device
                             // error; a non-finite row sets the non-finite bit
    bool pdl = true;         // with partials: launch as a programmatic dependent
    bool warp_units = false; // the partials come from warp units
};

cudaError_t launch_profile_select(const ProfileSelectArgs &a, cudaStream_t stream);

// fdllm_lmhead_select on the library-owned workspace, with programmatic dependent launches
// switched on or off (as select_owned).
fdllm_status lmhead_select_owned(const void *hidden, const void *w_vocab, int B, int L, int H,
                                 int V, uint8_t *mask, double param, int mode,
                                 int32_t *out_tokens, uint8_t *out_commit, int32_t *out_n,
                                 cudaStream_t stream, bool pdl);

// The library-owned workspace of the current device, at least `need` bytes.  Outside a capture it
// is grown to `reserve`, the most that any call of no larger a shape needs (where memory allows:
// a call goes on with `need`), and zero-filled when allocated; during one it stays as it is.
// Every user shares its 256-byte header: the sticky status word at offset 0 and the vocab
// reduction's work counter at 4 (zero between calls); the LM-head path keeps its compact row
// count at 8.
fdllm_status owned_workspace(size_t need, size_t reserve, cudaStream_t stream, void **out);

// Whether owned_workspace can give `need` bytes: the workspace holds them, or `stream` is not
// being captured (the workspace does not grow during a capture).
bool owned_workspace_ready(size_t need, cudaStream_t stream);

// The most workspace that any selection of no more and no longer rows needs; the need of an LM-head
// call, and the most of any with no more rows, no larger a hidden size and no longer a vocabulary.
size_t select_reserve_bytes(int64_t rows, int64_t row_bytes);
size_t lmhead_need_bytes(int64_t rows, int H, int V);
size_t lmhead_reserve_bytes(int64_t rows, int H, int V);

// fdllm_select's argument checks (shape, pointers, mode, param, logits alignment and the
// unit plan's index range), done before anything is enqueued.
fdllm_status check_select_args(const void *logits, int dtype, int B, int L, int V,
                               const uint8_t *mask, double param, int mode,
                               const int32_t *out_tokens, const uint8_t *out_commit,
                               const int32_t *out_n);

// Frees fdllm_select_host's device staging buffer of device `dev` (the caller synchronises).
void release_host_staging(int dev);

// fdllm_select on the library-owned workspace, with programmatic dependent launches
// switched on or off (the decode loop's graph body falls back to plain stream order where
// the driver does not accept programmatic edges inside a conditional node).
fdllm_status select_owned(const void *logits, int dtype, int B, int L, int V, uint8_t *mask,
                          double param, int mode, int32_t *out_tokens, uint8_t *out_commit,
                          int32_t *out_n, cudaStream_t stream, bool pdl);

struct ProfileTermsArgs {
    const float *conf;       // [B, L]
    const uint8_t *mask;     // [B, L]
    int B;
    int L;
    double *out_G;           // [B, L] by rank, nullable
    double *out_F;           // [B, L] by rank, nullable
    double *out_B;           // [B, L] by rank, nullable
    double delta;            // the profile rule's margin, for out_feff
    double *out_feff;        // [B, L] by rank: 1 - delta + B_n, nullable
    int32_t *out_order;      // [B, L] position at each rank, nullable
};

cudaError_t launch_profile_terms(const ProfileTermsArgs &a, cudaStream_t stream);

// ------------------------------------------------------------------ device helpers
#ifdef __CUDACC__
__device__ __forceinline__ float ex2_mufu(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Every partial (M, S) holds S = sum exp(x - M) relative to its own maximum M exactly.
//
// Sums are accumulated as 2^(x * s - r2) with a scale s and an fp32 reference r2.
//  * |ref| < kBigRef: s = log2e, r2 = round(ref * log2e).  The FMA forms x * log2e exactly;
//    the rounding residual r = ref * log2e - r2 is at most half an ulp of a value below 2^31,
//    so |r| <= 64, and it scales every term by the same 2^r, which rebase_scaled removes.
//  * |ref| >= kBigRef: s = 1, r2 = ref.  Distinct fp32 values there are at least 64 apart, so
//    every term but those equal to ref is below 2^-64 of them (under e^-64 in exp as well):
//    the sum counts the maxima, and the terms it drops weigh under 2^-40 for V < 2^24.
constexpr float kBigRef = 0x1p30f;

// S accumulated against (s, r2) -> relative to M: S * 2^(r2 - M s).  M s - r2 is formed in
// one FMA from the exact product, so the rounding of r2 cancels instead of scaling S.
__device__ __forceinline__ float rebase_scaled(float S, float s, float r2, float M)
{
    return S != 0.0f ? S * ex2_mufu(-fmaf(M, s, -r2)) : 0.0f;  // keeps NaN, avoids 0 * inf
}

// S relative to the maximum a -> relative to b >= a: S * exp(a - b).  a - b is exact when the
// two are within a factor of two and carries a relative 2^-24 otherwise, where the factor is
// below exp(-|b| / 2).  Infinite or NaN maxima give NaN, reported by the caller.
__device__ __forceinline__ float rebase(float S, float a, float b)
{
    return S != 0.0f ? S * ex2_mufu((a - b) * kLog2e) : 0.0f;
}

// Results of P positions from their units, folded in unit order, eight at a time (a fixed order,
// so identical rows give identical bits): c = min(1/S, 1) (the max term alone is 1) and x_hat =
// the first index attaining the max; c = NaN, x_hat = -1 when the row holds a NaN or its maximum
// is +inf or -inf.  p[i] is null for a position without partials (c and tok untouched).  The P
// positions' loads are in flight together.
template <int P>
__device__ __forceinline__ void combine_positions(const UnitPartial *const (&p)[P], int upr,
                                                  float (&c)[P], int32_t (&tok)[P])
{
    constexpr int U = 8;
    float M[P], S[P];
    uint32_t idx[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        M[i] = -__int_as_float(0x7F800000);
        S[i] = 0.0f;
        idx[i] = kNoIdx;
    }
    for (int j0 = 0; j0 < upr; j0 += U) {
        const int cnt = upr - j0 < U ? upr - j0 : U;
        float Mj[P][U], Sj[P][U];
        uint32_t Ij[P][U];
#pragma unroll
        for (int i = 0; i < P; ++i)
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (j < cnt && p[i] != nullptr) {
                    const int4 r = __ldcg(reinterpret_cast<const int4 *>(p[i] + j0 + j));
                    Mj[i][j] = __int_as_float(r.x);
                    Sj[i][j] = __int_as_float(r.y);
                    Ij[i][j] = (uint32_t)r.z;
                }
#pragma unroll
        for (int i = 0; i < P; ++i) {
            if (p[i] == nullptr)
                continue;
            float Mb = M[i];
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (j < cnt)
                    Mb = fmaxf(Mb, Mj[i][j]);
            float Sb = rebase(S[i], M[i], Mb);
            uint32_t ib = (M[i] == Mb) ? idx[i] : kNoIdx;
#pragma unroll
            for (int j = 0; j < U; ++j)
                if (j < cnt) {
                    Sb += rebase(Sj[i][j], Mj[i][j], Mb);
                    if (Mj[i][j] == Mb && ib == kNoIdx)
                        ib = Ij[i][j];
                }
            M[i] = Mb;
            S[i] = Sb;
            idx[i] = ib;
        }
    }
#pragma unroll
    for (int i = 0; i < P; ++i) {
        if (p[i] == nullptr)
            continue;
        const bool finite = fabsf(M[i]) <= 3.402823466e38f && fabsf(S[i]) <= 3.402823466e38f;
        const bool ok = finite && S[i] > 0.0f && idx[i] != kNoIdx;
        tok[i] = ok ? (int32_t)idx[i] : -1;
        c[i] = ok ? fminf(1.0f / S[i], 1.0f) : __int_as_float(0x7FC00000);
    }
}

__device__ __forceinline__ void combine_position(const UnitPartial *p, int upr, float &c,
                                                 int32_t &tok)
{
    const UnitPartial *const pp[1] = {p};
    float cc[1];
    int32_t tt[1];
    combine_positions(pp, upr, cc, tt);
    c = cc[0];
    tok = tt[0];
}

// Programmatic dependent launch: the dependent grid's wait for the primary grid's results,
// and the primary's permission for the dependent grid to start launching.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

}  // namespace fdllm
