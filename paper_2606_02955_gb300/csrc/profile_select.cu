// profile_select.cu -- steps a2-a5 of the selection for one batch row per CTA (paper
// Algorithm 1: sort, scan, select, reveal):
//   a2  sort the masked (c, position) pairs by c descending, position ascending, as 64-bit
//       keys; rows of at most 32 positions (one warp) by rank counting (each key's rank is the
//       number of smaller keys, 32 independent shuffles), longer rows by a bitonic network of
//       two keys per thread (shuffles and registers up to distance 32, shared memory above);
//   a3  prefix sums over the sorted order in 64-bit fixed point (units of 2^-52, exact and
//       independent of the summation order; warp shuffles, then across warps):
//       P_n = sum_{j<=n} (1 - c_(j)), so L_n = max{0, 1 - P_n} (= sum c - (n-1), Sec. 3),
//       U_n = 1 - c_(n), G_n = L_n - U_n; factor: (n+1)(1 - c_(n)) < f; threshold: c_(n) >= tau;
//   a4  n* = max{n : rule accepts n} (a block max, the literal definition), 1 if none;
//   a5  reveal the first n* sorted positions: token, commit flag, mask cleared.
// The row has L <= 1024 positions, so this is latency-bound work on a few KB: the kernel's
// time after its launch wait is the selection's share of a decode step.  No fp64
// arithmetic: GB300's fp64 pipe is slow enough (on the order of a hundred cycles per
// dependent operation) that an fp64 scan and rule cost more than the sort.
#include <cmath>
#include <cstdint>

#include "fdllm_internal.cuh"
#include "ptx.cuh"

namespace fdllm {
namespace {

constexpr uint64_t kPadKey = ~0ull;  // sorts after every real key

// Fixed point of the scan: 1 - c in units of 2^-52.  c is an fp32 value in [0, 1], so
// c * 2^52 is exact in fp32 and an integer for every c >= 2^-29; smaller c round to the
// nearest unit (an absolute error of at most 2^-53 per term).  A prefix of up to 1024 terms
// stays below 2^63, and integer addition makes the sums exact and order-independent.
constexpr int64_t kFixOne = (int64_t)1 << 52;

__device__ __forceinline__ int64_t one_minus_fixed(float c)
{
    return kFixOne - __float2ll_rn(c * 0x1p52f);
}

// Masked: (bits(1) - bits(c)) << 32 | pos — for c in [0, 1] larger c gives a smaller key
// (0 for c = 1, bits(1) for c = 0), and equal c falls back to the position.  Unmasked:
// 0xFFFFFFFF << 32 | pos, after every masked key.
constexpr uint32_t kOneBits = 0x3F800000u;

__device__ __forceinline__ uint64_t make_key(bool masked, float c, int pos)
{
    const uint32_t hi = masked ? kOneBits - __float_as_uint(c) : 0xFFFFFFFFu;
    return ((uint64_t)hi << 32) | (uint32_t)pos;
}

__device__ __forceinline__ float key_conf(uint64_t key)
{
    return __uint_as_float(kOneBits - (uint32_t)(key >> 32));
}

// Barrier of a row's W warps (the CTA may hold idle ones, see kSpreadThreads).
template <int W>
__device__ __forceinline__ void row_barrier()
{
    asm volatile("barrier.cta.sync 1, %0;" ::"n"(32 * W) : "memory");
}

// A row of more than 32 positions is held by W warps of K keys per thread: element
// (w K + r) 32 + lane is key[r] of that lane of warp w.
//
// Bitonic sort of the N = 32 K W keys.  Partners up to 16 apart are shuffled, 32 (and 64, with
// K = 4) apart are registers of one thread, and only those 32 K or more apart go through shared
// memory (two halves of buf[2 N] in turn, one barrier per stage).  What bounds the kernels is the
// latency of this chain and, after the vocab reduction, of the partials' loads, so the selection
// takes two keys per thread: four put two rounds of loads in a row (12.4 us after the reduction
// at L = 1024 and 5 units per row, two keys 8.9, one key 9.8 and, with the earlier one-key
// kernel's two barriers per stage, 11.7), and one key needs 15 shared stages for 1024 positions
// where two need 10.  On given confidences: 1000 positions 9.6 -> 6.6 us, 256 4.0 -> 3.3, 61 2.7
// -> 2.3.  The terms kernel loads one value per position: four keys at 1024 (14.8 -> 8.3 us; 9.2
// with two), two below (256 5.2 -> 3.7).
template <int W, int K>
__device__ __forceinline__ void sort_keys(uint64_t (&key)[K], uint64_t *buf)
{
    constexpr int N = 32 * K * W;
    const int lane = threadIdx.x & 31;
    const int idx0 = (int)(threadIdx.x >> 5) * 32 * K + lane;
    int turn = 0;  // the half of buf[2 N] in use
#pragma unroll 1
    for (int k = 2; k <= N; k <<= 1) {
        bool up[K];  // the element's run of k is sorted upwards
#pragma unroll
        for (int r = 0; r < K; ++r)
            up[r] = ((idx0 + 32 * r) & k) == 0;
        if constexpr (W > 1) {
#pragma unroll 1
            for (int j = k >> 1; j >= 32 * K; j >>= 1) {
#pragma unroll
                for (int r = 0; r < K; ++r)
                    buf[turn + idx0 + 32 * r] = key[r];
                row_barrier<W>();
#pragma unroll
                for (int r = 0; r < K; ++r) {
                    const uint64_t other = buf[turn + ((idx0 + 32 * r) ^ j)];
                    if ((other < key[r]) == (((idx0 & j) == 0) == up[r]))
                        key[r] = other;
                }
                turn = N - turn;
            }
        }
#pragma unroll
        for (int jr = K / 2; jr >= 1; jr >>= 1)
            if (k >= 64 * jr)
#pragma unroll
                for (int r = 0; r < K; ++r)
                    if ((r & jr) == 0 && (key[r + jr] < key[r]) == up[r]) {
                        const uint64_t t = key[r];
                        key[r] = key[r + jr];
                        key[r + jr] = t;
                    }
#pragma unroll 1
        for (int j = k >= 32 ? 16 : k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int r = 0; r < K; ++r) {
                const uint64_t other = __shfl_xor_sync(0xFFFFFFFFu, key[r], j);
                if ((other < key[r]) == (((lane & j) == 0) == up[r]))
                    key[r] = other;
            }
    }
}

// Inclusive prefix sums of v over the elements in order.
template <int W, int K, typename V>
__device__ __forceinline__ void scan_elements(V (&v)[K], V *warp_tot)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const V u = __shfl_up_sync(0xFFFFFFFFu, v[r], o);
            if (lane >= o)
                v[r] += u;
        }
    V base = V(0);
    if constexpr (W > 1) {
        V total = V(0);
#pragma unroll
        for (int r = 0; r < K; ++r)
            total += __shfl_sync(0xFFFFFFFFu, v[r], 31);
        if (lane == 0)
            warp_tot[w] = total;
        row_barrier<W>();
        for (int i = 0; i < w; ++i)
            base += warp_tot[i];
    }
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const V last = __shfl_sync(0xFFFFFFFFu, v[r], 31);
        v[r] += base;
        base += last;
    }
}

// The rule's acceptance of prefix size n, from c_(n) (fp32), v = 1 - c_(n) and the prefix
// P_n = sum_{j<=n} (1 - c_(j)) in fixed point.  `bound`: for the profile (and robust) rule
// delta = 1 - f in fixed point, for the factor rule f; `tau_f`: the smallest fp32 value
// >= tau, so that c >= tau_f in fp32 decides c >= tau exactly.
__device__ __forceinline__ bool rule_accepts(int mode, int n, float cn, int64_t v, int64_t P,
                                             int64_t bound, float tau_f)
{
    if (mode == 0 || mode == kModeRobust) {  // profile: G_n = L_n - U_n > delta
        const int64_t Ln = kFixOne - P > 0 ? kFixOne - P : 0;
        return Ln - v > bound;
    }
    if (mode == 1)  // factor: (n+1)(1 - c_(n)) < f
        return (int64_t)(n + 1) * v < bound;
    return cn >= tau_f;  // threshold: c_(n) >= tau
}

// Where rows' CTAs start while the kernel before them holds the SMs (the warp units all registers
// of every SM, the confidences' own pass many of its threads), small ones are all placed on the first
// few SMs to be freed, where their loads and sorts then queue.  CTAs of 512 threads, the warps
// beyond a row's own returning at once, spread over more.  Time over the reduction alone, a row's
// own warps against 512 threads: 64 x 32 positions of 32000 bf16 logits 7.8 -> 3.1 us, of 20000 5.0
// -> 2.6, 131 x 61 of 20008 fp16 7.5 -> 5.1, 64 x 256 of 16384 8.1 -> 4.9 (with 256 threads 3.2,
// 2.4, 5.1 and 7.0; with 1024 3.2, 2.4, 6.2 and 6.4).  After CTA units, which leave room for small
// CTAs beside them, it gains nothing (one row 7.3 against 7.5 us a step), nor with more than two
// CTAs per SM (1000 x 32 positions 41.9 against 42.1).
constexpr int kSpreadThreads = 512;
constexpr int kSpreadCtas = 2 * 152;
// The terms kernel's CTAs have 1024 threads: after 63 x 1000 confidences of 1004 logits their share
// of a call 32.5 us with a row's own 256, 17.2 with 512, 10.9 with 1024; 64 x 256 8.2, 5.5 and 4.4.
constexpr int kSpreadTerms = 1024;

bool spread_rows(int64_t ctas) { return ctas > 4 && ctas <= kSpreadCtas; }

template <int W, int K>
__global__ void __launch_bounds__(kSpreadThreads)
    profile_select_kernel(const ProfileSelectArgs a, int64_t bound, float tau_f)
{
    static_assert(32 * W <= kSpreadThreads, "a row's warps");
    if (threadIdx.x >= 32 * W)
        return;
    constexpr int N = 32 * K * W;
    __shared__ uint64_t sk[W > 1 ? 2 * N : 1];
    __shared__ int32_t s_tok[N];
    __shared__ int64_t warp_tot[W];
    __shared__ int warp_m[W], warp_n[W];
    constexpr unsigned kFull = 0xFFFFFFFFu;

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int pos0 = w * 32 * K + lane;  // this thread's positions: pos0 + 32 r
    const int L = a.L;
    const int64_t base = (int64_t)blockIdx.x * L;

    // (c, x_hat) of this thread's positions: folded from the vocab reduction's unit
    // partials, or read from the given arrays.  Launched as a programmatic dependent: the
    // producer of the partials or confidences has completed past the launch wait.  As in the
    // warp kernel, after the vocab reduction the mask bytes and the allowances are loaded
    // before that wait (their writers completed before the reduction passed its own wait,
    // and the reduction writes neither); the partials or confidences and the status word
    // after it, all issued before any is used.
    const bool early = a.partials != nullptr;
    uint8_t mask_byte[K];
    float eta[K];
    auto load_row_inputs = [&]() {
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int pos = pos0 + 32 * r;
            mask_byte[r] = pos < L ? __ldcg(a.mask + base + pos) : (uint8_t)0;
            eta[r] = (float)a.eta;
            if (a.mode == kModeRobust && a.eta_pos != nullptr && pos < L)
                eta[r] = fmaxf(__ldcg(a.eta_pos + base + pos), 0.0f);  // negative or NaN: 0
        }
    };
    if (threadIdx.x == 0)
        pdl_launch_dependents();  // a following vocab reduction may start its prologue
    if (early)
        load_row_inputs();
    pdl_wait();
    if (!early)
        load_row_inputs();
    const bool dev_err = a.status != nullptr && (__ldcg(a.status) & kDevStatTimeout) != 0;
    float c[K];
    int32_t tok[K];
    if (a.partials != nullptr) {
        const int upr = a.units_per_row;
        const UnitPartial *p[K];
#pragma unroll
        for (int r = 0; r < K; ++r)  // unmasked positions have none
            p[r] = mask_byte[r] != 0 ? a.partials + (base + pos0 + 32 * r) * upr : nullptr;
        combine_positions(p, upr, c, tok);
    } else {
#pragma unroll
        for (int r = 0; r < K; ++r)
            if (pos0 + 32 * r < L) {
                c[r] = __ldcg(a.conf + base + pos0 + 32 * r);
                tok[r] = __ldcg(a.tok + base + pos0 + 32 * r);
            }
    }
    if (a.partials != nullptr && a.next_unit != nullptr && blockIdx.x == 0 && threadIdx.x == 0)
        *a.next_unit = 0;  // the vocab reduction before this kernel has finished
    uint64_t key[K];
    int m = 0;
    bool any_bad = false;
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int pos = pos0 + 32 * r;
        const bool masked = mask_byte[r] != 0;
        if (!masked) {
            c[r] = 0.0f;
            tok[r] = -1;
        }
        s_tok[pos] = tok[r];
        const bool bad = masked && !(c[r] > 0.0f && c[r] <= 1.0f);  // NaN fails both
        // The robust rule ranks and scans lower confidences max{0, c - eta} (App. C).
        float c_rank = c[r];
        if (a.mode == kModeRobust && masked && !bad)
            c_rank = fmaxf(0.0f, c[r] - eta[r]);
        key[r] = pos < L ? make_key(masked, c_rank, pos) : kPadKey;
        m += __popc(__ballot_sync(kFull, masked));
        any_bad |= __any_sync(kFull, bad) != 0;
    }
    if constexpr (W > 1) {
        if (lane == 0)
            warp_m[w] = any_bad ? -1 : m;
        row_barrier<W>();
        m = 0;
        any_bad = false;
#pragma unroll
        for (int i = 0; i < W; ++i) {
            any_bad |= warp_m[i] < 0;
            m += warp_m[i];  // meaningless, and unused, with a bad position
        }
    } else {
        __syncwarp();
    }

    sort_keys<W, K>(key, sk);

    // This thread now holds, as key[r], the n-th most confident masked position when n <= m.
    int64_t v[K], P[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        v[r] = pos0 + 32 * r < m ? one_minus_fixed(key_conf(key[r])) : 0;
        P[r] = v[r];
    }
    scan_elements<W, K>(P, warp_tot);
    int nstar = 0;
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int n = pos0 + 32 * r + 1;
        if (n <= m && rule_accepts(a.mode, n, key_conf(key[r]), v[r], P[r], bound, tau_f))
            nstar = n;  // n grows with r
    }
    nstar = __reduce_max_sync(kFull, nstar);
    if constexpr (W > 1) {
        if (lane == 0)
            warp_n[w] = nstar;
        row_barrier<W>();
#pragma unroll
        for (int i = 0; i < W; ++i)
            nstar = max(nstar, warp_n[i]);
    }
    if (m > 0 && nstar == 0)
        nstar = 1;  // progress convention
    if (any_bad) {
        nstar = -1;
        if (threadIdx.x == 0 && a.status != nullptr)
            atomicOr(a.status, kDevStatNonfinite);
    }
    if (dev_err)
        nstar = -2;

#pragma unroll
    for (int r = 0; r < K; ++r)
        if (pos0 + 32 * r < L) {
            const int pos = (int)(key[r] & 0xFFFFFFFFu);
            const bool commit = pos0 + 32 * r < nstar;  // nstar <= m: only masked keys qualify
            a.out_commit[base + pos] = commit ? 1 : 0;
            if (commit) {
                a.out_tokens[base + pos] = s_tok[pos];
                a.mask[base + pos] = 0;
            }
        }
    if (threadIdx.x == 0)
        a.out_n[blockIdx.x] = nstar;
}

// The same steps for rows of at most 32 positions, one warp per row: no block barriers, the
// sort by rank counting (the keys are distinct: the position is in their low bits, pads
// included), the scan by warp shuffles alone.  More than two rows per SM go kWarpRows to a CTA:
// CTAs of one row start at about one per ns (65536 rows of one position 101 -> 70 us a step, 2048 x 32
// positions 51.1 -> 50.3, 305 x 32 19.4 -> 18.6).
constexpr int kWarpRows = 8;

__global__ void __launch_bounds__(kSpreadThreads)
    profile_select_warp_kernel(const ProfileSelectArgs a, int rows_per_cta, int64_t bound,
                               float tau_f)
{
    __shared__ uint64_t s_keys[kWarpRows][32];
    __shared__ int32_t s_toks[kWarpRows][32];
    constexpr unsigned kFull = 0xFFFFFFFFu;
    const int t = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t row = (int64_t)blockIdx.x * rows_per_cta + w;
    if (w >= rows_per_cta || row >= a.B)
        return;
    uint64_t *const sk = s_keys[w];
    int32_t *const s_tok = s_toks[w];
    const int L = a.L;
    const int64_t base = row * L;

    // After the vocab reduction (partials given), the mask byte and the allowance are loaded
    // before the launch wait: this kernel starts only once the reduction has passed its own
    // launch wait, so whatever wrote them has completed, and the reduction writes neither.
    // The unit partials and the status word are the reduction's output: loaded after it.
    // Otherwise (confidences given) everything is loaded after the wait.
    const bool in_row = t < L;
    const bool early = a.partials != nullptr;
    uint8_t mask_byte = 0;
    float eta = (float)a.eta;
    auto load_row_inputs = [&]() {
        mask_byte = in_row ? __ldcg(a.mask + base + t) : (uint8_t)0;
        if (a.mode == kModeRobust && a.eta_pos != nullptr && in_row)
            eta = fmaxf(__ldcg(a.eta_pos + base + t), 0.0f);  // negative or NaN: 0
    };
    if (t == 0)
        pdl_launch_dependents();  // a following vocab reduction may start its prologue
    if (early)
        load_row_inputs();
    pdl_wait();  // the producer of the partials or confidences has completed
    if (!early)
        load_row_inputs();
    // The rest of the row's loads are issued here, before any of them is used (one memory
    // round trip): status word and the position's unit partials or (c, x_hat).
    const uint32_t status = a.status != nullptr ? __ldcg(a.status) : 0u;
    const bool masked = mask_byte != 0;
    float c = 0.0f;
    int32_t tok = -1;
    if (in_row && (masked || !early)) {  // unmasked positions have no partials
        if (early) {
            combine_position(a.partials + (base + t) * a.units_per_row, a.units_per_row, c,
                             tok);
        } else {
            c = __ldcg(a.conf + base + t);
            tok = __ldcg(a.tok + base + t);
        }
    }
    if (!masked) {
        c = 0.0f;
        tok = -1;
    }
    s_tok[t] = tok;
    if (a.partials != nullptr && a.next_unit != nullptr && row == 0 && t == 0)
        *a.next_unit = 0;  // the vocab reduction before this kernel has finished
    const bool bad = masked && !(c > 0.0f && c <= 1.0f);  // NaN fails both
    float c_rank = c;
    if (a.mode == kModeRobust && masked && !bad)
        c_rank = fmaxf(0.0f, c - eta);  // App. C: lower confidences max{0, c - eta}
    uint64_t key = make_key(masked, c_rank, t);
    const int m = __popc(__ballot_sync(kFull, masked));
    const bool any_bad = __any_sync(kFull, bad);

    int rank = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j)
        rank += __shfl_sync(kFull, key, j) < key ? 1 : 0;
    sk[rank] = key;
    __syncwarp();
    key = sk[t];

    // Lane t now holds the (t+1)-th most confident masked position when t < m.
    const int n = t + 1;
    const bool live = t < m;
    const float cn = live ? key_conf(key) : 1.0f;
    const int64_t v = live ? one_minus_fixed(cn) : 0;
    int64_t P = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(kFull, P, o);
        if (t >= o)
            P += u;
    }
    const bool ok = live && rule_accepts(a.mode, n, cn, v, P, bound, tau_f);
    int nstar = __reduce_max_sync(kFull, ok ? n : 0);
    if (m > 0 && nstar == 0)
        nstar = 1;  // progress convention
    if (any_bad) {
        nstar = -1;
        if (t == 0 && a.status != nullptr)
            atomicOr(a.status, kDevStatNonfinite);
    }
    if ((status & kDevStatTimeout) != 0)
        nstar = -2;

    if (t < L) {
        const int pos = (int)(key & 0xFFFFFFFFu);  // < L: the L row keys precede the pads
        const bool commit = t < nstar;
        a.out_commit[base + pos] = commit ? 1 : 0;
        if (commit) {
            a.out_tokens[base + pos] = s_tok[pos];
            a.mask[base + pos] = 0;
        }
    }
    if (t == 0)
        a.out_n[row] = nstar;
}

// Heterogeneity-bonus diagnostics of one batch row per CTA (Prop. heterogeneity-bonus,
// Eq. heterogeneity_decomp): the masked confidences sorted as in the selection, an fp64
// inclusive scan S_n = sum_{j<=n} c_(j), and at rank n: G_n = max{0, S_n - (n-1)} - (1 - c_(n)),
// F_n = (n+1) c_(n) - n and B_n = S_n - n c_(n) (= sum_{j<n} (c_(j) - c_(n))); and the
// effective factor f_eff(n) = 1 - delta + B_n of Remark adaptive-factor.
template <int W, int K>
__global__ void __launch_bounds__(kSpreadTerms) profile_terms_kernel(const ProfileTermsArgs a)
{
    if (threadIdx.x >= 32 * W)
        return;
    constexpr int N = 32 * K * W;
    __shared__ uint64_t sk[W > 1 ? 2 * N : 1];
    __shared__ double warp_tot[W];
    __shared__ int warp_m[W];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int pos0 = w * 32 * K + lane;
    const int L = a.L;
    const int64_t base = (int64_t)blockIdx.x * L;
    pdl_wait();  // the confidences and the mask are written
    if (threadIdx.x == 0)
        pdl_launch_dependents();
    uint64_t key[K];
    int m = 0;
    uint8_t mask_byte[K];
    float c[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int pos = pos0 + 32 * r;
        mask_byte[r] = pos < L ? a.mask[base + pos] : (uint8_t)0;
        c[r] = pos < L ? a.conf[base + pos] : 0.0f;
    }
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int pos = pos0 + 32 * r;
        const bool masked = mask_byte[r] != 0;
        key[r] = pos < L ? make_key(masked, masked ? c[r] : 0.0f, pos) : kPadKey;
        m += __popc(__ballot_sync(0xFFFFFFFFu, masked));
    }
    if constexpr (W > 1) {
        if (lane == 0)
            warp_m[w] = m;
        row_barrier<W>();
        m = 0;
#pragma unroll
        for (int i = 0; i < W; ++i)
            m += warp_m[i];
    }
    sort_keys<W, K>(key, sk);
    double cn[K], S[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        cn[r] = pos0 + 32 * r < m ? (double)key_conf(key[r]) : 0.0;
        S[r] = cn[r];
    }
    scan_elements<W, K>(S, warp_tot);
    const double nan = __longlong_as_double(0x7FF8000000000000ll);
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int t = pos0 + 32 * r;
        if (t >= L)
            continue;
        const bool live = t < m;
        double G = nan, F = nan, Bn = nan, fe = nan;
        if (live) {  // fp64 runs at two lanes per clock and SM: none for the ranks past m
            const double n = (double)(t + 1);
            G = fmax(0.0, S[r] - (n - 1.0)) - (1.0 - cn[r]);
            F = (n + 1.0) * cn[r] - n;
            Bn = S[r] - n * cn[r];
            fe = 1.0 - a.delta + Bn;
        }
        if (a.out_G != nullptr)
            a.out_G[base + t] = G;
        if (a.out_F != nullptr)
            a.out_F[base + t] = F;
        if (a.out_B != nullptr)
            a.out_B[base + t] = Bn;
        if (a.out_feff != nullptr)
            a.out_feff[base + t] = fe;
        if (a.out_order != nullptr)
            a.out_order[base + t] = live ? (int32_t)(key[r] & 0xFFFFFFFFu) : -1;
    }
}

template <int W, int K>
cudaError_t launch_terms_t(const ProfileTermsArgs &a, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.B);
    cfg.blockDim = dim3(spread_rows(a.B) ? kSpreadTerms : 32 * W);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, profile_terms_kernel<W, K>, a);
}

template <typename Kernel, typename... Args>
cudaError_t launch_select(Kernel kern, int64_t ctas, int threads, const ProfileSelectArgs &a,
                          cudaStream_t stream, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(threads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.pdl ? 1 : 0;  // a programmatic dependent of the previous kernel
    return cudaLaunchKernelEx(&cfg, kern, a, args...);
}

// One CTA per row of W warps.
template <int W, int K>
cudaError_t launch_rows(const ProfileSelectArgs &a, bool spread, int64_t bound, float tau_f,
                        cudaStream_t stream)
{
    return launch_select(profile_select_kernel<W, K>, a.B, spread ? kSpreadThreads : 32 * W, a,
                         stream, bound, tau_f);
}

}  // namespace

cudaError_t launch_profile_select(const ProfileSelectArgs &a, cudaStream_t stream)
{
    // The rule's parameter in the kernels' arithmetic.  f in fixed point (clamped to
    // [-1500, 1500]: beyond, (n+1)(1 - c) <= 1025 decides every n the same way), and the
    // profile margin delta = 1 - f from the same integer, so that delta + f = 1 exactly and
    // the equal-confidence reduction to the factor rule holds bit for bit.
    const double f = a.param < -1500.0 ? -1500.0 : (a.param > 1500.0 ? 1500.0 : a.param);
    const int64_t f_fix = std::llround(f * 0x1p52);
    const int64_t bound = a.mode == 1 ? f_fix : kFixOne - f_fix;
    float tau_f = (float)a.param;  // the smallest fp32 value >= tau
    if ((double)tau_f < a.param)
        tau_f = std::nextafter(tau_f, INFINITY);
    const int per = a.L <= 32 && a.B > kSpreadCtas ? kWarpRows : 1;
    const int64_t ctas = (a.B + per - 1) / per;
    const bool room = a.partials != nullptr && !a.warp_units;  // after CTA units
    const bool spread = !room && spread_rows(ctas);
    if (a.L <= 32)
        return launch_select(profile_select_warp_kernel, ctas, spread ? kSpreadThreads : 32 * per,
                             a, stream, per, bound, tau_f);
    if (a.L <= 64)
        return launch_rows<1, 2>(a, spread, bound, tau_f, stream);
    if (a.L <= 128)
        return launch_rows<2, 2>(a, spread, bound, tau_f, stream);
    if (a.L <= 256)
        return launch_rows<4, 2>(a, spread, bound, tau_f, stream);
    if (a.L <= 512)
        return launch_rows<8, 2>(a, spread, bound, tau_f, stream);
    return launch_rows<16, 2>(a, spread, bound, tau_f, stream);
}

cudaError_t launch_profile_terms(const ProfileTermsArgs &a, cudaStream_t stream)
{
    if (a.L <= 32)
        return launch_terms_t<1, 1>(a, stream);
    if (a.L <= 64)
        return launch_terms_t<1, 2>(a, stream);
    if (a.L <= 128)
        return launch_terms_t<2, 2>(a, stream);
    if (a.L <= 256)
        return launch_terms_t<4, 2>(a, stream);
    if (a.L <= 512)
        return launch_terms_t<8, 2>(a, stream);
    return launch_terms_t<8, 4>(a, stream);
}

}  // namespace fdllm
