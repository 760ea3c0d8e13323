// host_io.cu -- the end-to-end path on host buffers: the rows of masked positions are read
// by the GPU straight from page-locked host memory (over the host link) into a device buffer,
// so that only the logits the selection needs cross the link; fdllm_select_host wraps that,
// the step and the copies of its results back to the host in one call.
#include <cuda_runtime.h>
#include <unistd.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "fdllm.h"
#include "fdllm_internal.cuh"
#include "host_view.h"

namespace fdllm {
namespace {

// Bound by the host link (210 GB/s), which takes about 0.4 MB in flight to fill: with few rows a
// row is cut into parts of at least 16 KB (one round of a CTA's loads), so that a few masked rows
// fill it too.  One CTA per row against parts, fdllm_select_host on 32 positions of LLaDA's
// vocabulary: 5 % masked 43.5 -> 36 us, 15 % 47.5 -> 39.8, 50 % 52.2 -> 46.5.  The most CTAs: at
// 8 x 32 positions, 4 parts a row (8 CTAs per SM) took 197 us, one part 195.4.
constexpr int64_t kGatherPartVecs = 1024;
constexpr int64_t kGatherCtas = 2 * 152;

// Copies the 16-byte vectors of the masked (b, l) rows: row blockIdx.x, the part_vecs vectors of
// part blockIdx.y.
__global__ void __launch_bounds__(256)
    gather_masked_rows_kernel(const int4 *src, int4 *dst, const uint8_t *mask,
                              int64_t vec_per_row, int64_t part_vecs)
{
    pdl_wait();  // the mask's writer has completed
    if (threadIdx.x == 0)
        pdl_launch_dependents();  // the vocab reduction may start its prologue
    const int64_t row = blockIdx.x;
    if (mask[row] == 0)
        return;
    const int64_t begin = blockIdx.y * part_vecs;
    const int64_t n = min(part_vecs, vec_per_row - begin);
    const int4 *s = src + row * vec_per_row + begin;
    int4 *d = dst + row * vec_per_row + begin;
    int64_t i = threadIdx.x;
    // Four loads in flight per thread: each crosses the host link with its full latency.
    for (; i + 3 * 256 < n; i += 4 * 256) {
        const int4 a = s[i], b = s[i + 256], c = s[i + 512], e = s[i + 768];
        d[i] = a;
        d[i + 256] = b;
        d[i + 512] = c;
        d[i + 768] = e;
    }
    for (; i < n; i += 256)
        d[i] = s[i];
}

// Where the GPU reads `src`: device memory as it is, page-locked host memory through its
// mapping; nullptr for pageable host memory (or an address CUDA does not know).
const void *device_view(const void *src)
{
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, src) != cudaSuccess) {
        (void)cudaGetLastError();
        return nullptr;
    }
    if (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged)
        return src;
    if (attr.type == cudaMemoryTypeHost)
        return attr.devicePointer;
    return nullptr;
}

// The mapping through which the GPU writes n elements of page-locked host memory; nullptr for any
// other memory and where a part of the array is not mapped.
template <typename T>
T *pinned_view(T *p, int64_t n)
{
    static const int64_t page = sysconf(_SC_PAGESIZE);
    auto device_of = [](uint8_t *host) -> uint8_t * {
        cudaPointerAttributes attr;
        if (cudaPointerGetAttributes(&attr, host) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        return attr.type == cudaMemoryTypeHost ? static_cast<uint8_t *>(attr.devicePointer)
                                               : nullptr;
    };
    return reinterpret_cast<T *>(whole_view(reinterpret_cast<uint8_t *>(p),
                                            n * (int64_t)sizeof(T), page, device_of));
}

// Whether the host itself reads and writes p (pageable or page-locked memory).
bool on_host(const void *p)
{
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return true;
    }
    return attr.type == cudaMemoryTypeUnregistered || attr.type == cudaMemoryTypeHost;
}

cudaError_t launch_gather(const void *dsrc, void *dst, const uint8_t *mask, int64_t rows,
                          int64_t row_bytes, cudaStream_t stream)
{
    const int64_t vecs = row_bytes / 16;
    const int64_t most = std::max<int64_t>(1, kGatherCtas / rows);
    const int64_t want = std::min((vecs + kGatherPartVecs - 1) / kGatherPartVecs, most);
    const int64_t part_vecs = (vecs + want - 1) / want;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)rows, (unsigned)((vecs + part_vecs - 1) / part_vecs));
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gather_masked_rows_kernel, static_cast<const int4 *>(dsrc),
                              static_cast<int4 *>(dst), mask, vecs, part_vecs);
}

// fdllm_select_host's device staging, one buffer per device, grown on demand (allocated
// outside the step's kernels, like the library workspace).
struct Staging {
    void *ptr = nullptr;
    size_t bytes = 0;
};
constexpr int kStageDevices = 64;
Staging g_stage[kStageDevices];
std::mutex g_stage_mutex;

size_t up256(size_t x) { return (x + 255) / 256 * 256; }

fdllm_status staging_buffer(size_t need, void **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kStageDevices)
        return FDLLM_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_stage_mutex);
    Staging &s = g_stage[dev];
    if (s.bytes < need) {
        if (s.ptr) {
            if (cudaDeviceSynchronize() != cudaSuccess)
                return FDLLM_ERR_CUDA;
            cudaFree(s.ptr);
            s.ptr = nullptr;
            s.bytes = 0;
        }
        void *p = nullptr;
        if (cudaMalloc(&p, need) != cudaSuccess)
            return FDLLM_ERR_CUDA;
        s.ptr = p;
        s.bytes = need;
    }
    *out = s.ptr;
    return FDLLM_OK;
}

}  // namespace

void release_host_staging(int dev)
{
    if (dev < 0 || dev >= kStageDevices)
        return;
    std::lock_guard<std::mutex> lock(g_stage_mutex);
    if (g_stage[dev].ptr) {
        cudaDeviceSynchronize();
        cudaFree(g_stage[dev].ptr);
        g_stage[dev].ptr = nullptr;
        g_stage[dev].bytes = 0;
    }
}

}  // namespace fdllm

using namespace fdllm;

extern "C" fdllm_status fdllm_gather_masked_rows(const void *src, void *dst, int dtype, int B,
                                                 int L, int V, const uint8_t *mask, void *stream)
{
    if (!src || !dst || !mask || B < 1 || L < 1 || L > FDLLM_MAX_L || V < 1 ||
        (int64_t)B * L > FDLLM_MAX_ROWS ||
        (dtype != FDLLM_BF16 && dtype != FDLLM_FP32 && dtype != FDLLM_FP16))
        return FDLLM_ERR_ARG;
    const int64_t row_bytes = (int64_t)V * (dtype == FDLLM_FP32 ? 4 : 2);
    if (row_bytes % 16 != 0 || (reinterpret_cast<uintptr_t>(src) & 15u) ||
        (reinterpret_cast<uintptr_t>(dst) & 15u))
        return FDLLM_ERR_ALIGN;
    // The device-side address of src: page-locked host memory is read through its mapping.
    const void *dsrc = device_view(src);
    if (!dsrc || (reinterpret_cast<uintptr_t>(dsrc) & 15u))
        return FDLLM_ERR_ARG;  // pageable host memory: not readable by the GPU here
    return launch_gather(dsrc, dst, mask, (int64_t)B * L, row_bytes,
                         static_cast<cudaStream_t>(stream)) == cudaSuccess
               ? FDLLM_OK
               : FDLLM_ERR_CUDA;
}

extern "C" fdllm_status fdllm_select_host(const void *logits, int dtype, int B, int L, int V,
                                          uint8_t *mask, double param, int mode,
                                          int32_t *out_tokens, uint8_t *out_commit,
                                          int32_t *out_n, void *stream)
{
    fdllm_status st = check_select_args(logits, dtype, B, L, V, mask, param, mode, out_tokens,
                                        out_commit, out_n);
    if (st != FDLLM_OK)
        return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t rows = (int64_t)B * L;
    const int64_t row_bytes = (int64_t)V * (dtype == FDLLM_FP32 ? 4 : 2);
    // Logits already in device memory are read in place; page-locked host logits are read
    // by the GPU at the masked rows only; pageable host logits are copied whole.
    cudaPointerAttributes attr;
    const bool known = cudaPointerGetAttributes(&attr, logits) == cudaSuccess;
    if (!known)
        (void)cudaGetLastError();
    const bool on_device =
        known && (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged);
    const void *mapped = known && attr.type == cudaMemoryTypeHost ? attr.devicePointer : nullptr;
    const size_t logits_bytes = on_device ? 0 : up256((size_t)(rows * row_bytes));
    const size_t off_mask = logits_bytes;
    const size_t off_tok = off_mask + up256((size_t)rows);
    const size_t off_commit = off_tok + up256((size_t)rows * 4);
    const size_t off_n = off_commit + up256((size_t)rows);
    const size_t total = off_n + up256((size_t)B * 4);
    void *stage = nullptr;
    st = staging_buffer(total, &stage);
    if (st != FDLLM_OK)
        return st;
    uint8_t *base = static_cast<uint8_t *>(stage);
    uint8_t *d_mask = base + off_mask;
    // Page-locked results are written in place by the selection, over the host link, and the
    // host clears the committed positions of its own mask afterwards: one copy (the mask in)
    // instead of six, each of which held the stream for 1.5 to 3 us (8 x 32 positions of LLaDA's
    // vocabulary 208 -> 195 us a call, 32 short rows 44 -> 33, 64 x 1024 271 -> 263).
    int32_t *v_tok = nullptr, *v_n = nullptr;
    uint8_t *v_commit = nullptr;
    if (on_host(mask)) {
        v_tok = pinned_view(out_tokens, rows);
        v_commit = pinned_view(out_commit, rows);
        v_n = pinned_view(out_n, B);
    }
    const bool in_place = v_tok && v_n && v_commit;
    int32_t *d_tok = in_place ? v_tok : reinterpret_cast<int32_t *>(base + off_tok);
    uint8_t *d_commit = in_place ? v_commit : base + off_commit;
    int32_t *d_n = in_place ? v_n : reinterpret_cast<int32_t *>(base + off_n);
    const void *d_logits = on_device ? logits : base;

    // Inputs: the mask, the caller's token array where it is staged (the step writes only
    // committed positions, the others keep the caller's values), then the logits the step reads.
    if (cudaMemcpyAsync(d_mask, mask, (size_t)rows, cudaMemcpyDefault, s) != cudaSuccess ||
        (!in_place && cudaMemcpyAsync(d_tok, out_tokens, (size_t)rows * 4, cudaMemcpyDefault,
                                      s) != cudaSuccess))
        return FDLLM_ERR_CUDA;
    if (!on_device) {
        if (mapped && (reinterpret_cast<uintptr_t>(mapped) & 15u) == 0) {
            if (launch_gather(mapped, base, d_mask, rows, row_bytes, s) != cudaSuccess)
                return FDLLM_ERR_CUDA;
        } else if (cudaMemcpyAsync(base, logits, (size_t)(rows * row_bytes), cudaMemcpyDefault,
                                   s) != cudaSuccess) {
            return FDLLM_ERR_CUDA;
        }
    }
    st = select_owned(d_logits, dtype, B, L, V, d_mask, param, mode, d_tok, d_commit, d_n, s,
                      true);
    if (st != FDLLM_OK)
        return st;
    if (in_place) {
        if (cudaStreamSynchronize(s) != cudaSuccess)
            return FDLLM_ERR_CUDA;
        for (int64_t i = 0; i < rows; ++i)
            mask[i] = out_commit[i] ? 0 : mask[i];
        return FDLLM_OK;
    }
    if (cudaMemcpyAsync(out_tokens, d_tok, (size_t)rows * 4, cudaMemcpyDefault, s) !=
            cudaSuccess ||
        cudaMemcpyAsync(out_commit, d_commit, (size_t)rows, cudaMemcpyDefault, s) !=
            cudaSuccess ||
        cudaMemcpyAsync(out_n, d_n, (size_t)B * 4, cudaMemcpyDefault, s) != cudaSuccess ||
        cudaMemcpyAsync(mask, d_mask, (size_t)rows, cudaMemcpyDefault, s) != cudaSuccess)
        return FDLLM_ERR_CUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? FDLLM_OK : FDLLM_ERR_CUDA;
}
