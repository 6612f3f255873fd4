// Trap handler data path (paper Section 5.4): while a sequence waits for an interrupt its KV cache can
// be swapped to host memory and brought back later, possibly into other pages.  The swapped form of a
// sequence is its pages in logical order, one contiguous image [n_pages][2][Hkv][16][d].
//
// Swap-out gathers the pages into a contiguous device staging buffer with one kernel and then moves
// the image to (pinned) host memory with ONE asynchronous copy, so that PCIe sees a single long
// transfer instead of one per page; swap-in is the mirror image.  A small image in page-locked memory is
// written and read by the kernel itself.  The keep / swap / recompute rule of
// the same section is evaluated on the host by asynclm_trap_decide.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "asynclm.h"
#include "common.cuh"
#include "kernels.h"

namespace asynclm {

// Page ids as the kernel gets them: in its parameters, which saves a copy in the stream in front of it, or in device memory.
constexpr int kIdsInParams = 960;
struct IdsByValue {
    int32_t id[kIdsInParams];
    __device__ __forceinline__ int32_t operator[](int64_t k) const { return id[k]; }
};
struct IdsInMemory {
    const int32_t* id;
    __device__ __forceinline__ int32_t operator[](int64_t k) const { return __ldg(id + k); }
};

// A page is one contiguous run of `vpp` 16-byte vectors in the pool; page j of the image is page ids[j]
// of the pool.  Four vectors in flight per thread; consecutive threads take consecutive vectors.  HOST: the image is
// page-locked host memory, read past the caches.
template <bool TO_POOL, bool HOST, typename Ids>
__global__ void __launch_bounds__(256)
page_copy_kernel(uint4* __restrict__ pool, uint4* __restrict__ image, const __grid_constant__ Ids ids,
                 int64_t total, int vpp) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < total; i0 += 4 * stride) {
        uint4 v[4];
        int64_t at[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = i0 + u * stride;
            at[u] = -1;
            if (i < total) {
                at[u] = (int64_t)ids[i / vpp] * vpp + i % vpp;
                if constexpr (!TO_POOL) v[u] = ldg_nc_v4(pool + at[u]);
                else if constexpr (HOST) v[u] = ld_host_v4(image + i);
                else v[u] = ldg_nc_v4(image + i);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = i0 + u * stride;
            if (at[u] >= 0) {
                if (TO_POOL) pool[at[u]] = v[u];
                else image[i] = v[u];
            }
        }
    }
}

static size_t page_bytes(const asynclm_shape* s) {
    return (size_t)2 * s->num_kv_heads * s->page_size * s->head_dim * 2;
}

static int check_swap_args(const asynclm_shape* s, const int32_t* ids, int32_t n, const void* pool, const void* staging,
                           const void* host_image, bool distinct) {
    if (!s || s->num_kv_heads <= 0 || s->page_size <= 0 || s->head_dim <= 0 || s->head_dim % 8 != 0 || n < 0)
        return ASYNCLM_ERR_INVALID_ARG;
    if (n == 0) return ASYNCLM_OK;
    if (!ids || !pool || !staging || !host_image || (((uintptr_t)pool | (uintptr_t)staging | (uintptr_t)host_image) & 15) != 0)
        return ASYNCLM_ERR_INVALID_ARG;
    for (int32_t j = 0; j < n; ++j)
        if (ids[j] < 0 || ids[j] >= s->num_pages) return ASYNCLM_ERR_PAGE_TABLE;
    if (distinct) {
        std::vector<int32_t> sorted(ids, ids + n);
        std::sort(sorted.begin(), sorted.end());
        if (std::adjacent_find(sorted.begin(), sorted.end()) != sorted.end()) return ASYNCLM_ERR_PAGE_TABLE;
    }
    return ASYNCLM_OK;
}

// What bounds a small swap is the copies' latency: each waits for what is in front of it to be flushed and the next one waits for it.
// So up to kIdsInParams page ids (what 4 KB of parameters hold) go as parameters instead of by a copy, and an image of up to kDirectBytes that is
// page-locked is read or written by the kernel in place.  us out + in, before | now, back to back: 28 KB 27.8 | 16.6, 256 KB 42.0 |
// 23.7, 512 KB 51.5 | 32.8, 1 MB 68 | 54, 2 MB 108 | 94; one call alone up to 10 less, at 2 MB the same.  The line lies where the bus
// takes the time and the copy engine leaves the SMs to other streams: 32 CTAs keep the bus busy as well as more do.  Larger: 4 MB 183 | 177, 32 MB 1244 |
// 1230.  More ids in pieces of 960, a kernel each, lost to their one copy: 8000 pages of 4 KB 604 | 620.
constexpr size_t kDirectBytes = 2 << 20;
constexpr int kDirectCtas = 32;

template <bool TO_POOL, bool HOST, typename Ids>
static int copy_pages(const void* pool, void* image, const Ids& ids, int64_t total, int vpp, cudaStream_t s) {
    const int64_t blocks = std::min<int64_t>((total + 4 * 256 - 1) / (4 * 256), HOST ? kDirectCtas : 148 * 8);
    page_copy_kernel<TO_POOL, HOST><<<(int)blocks, 256, 0, s>>>((uint4*)const_cast<void*>(pool), (uint4*)image, ids, total, vpp);
    return cuda_status(cudaGetLastError());
}

// A copy in a graph reads ids and image when the graph runs, parameters are taken now: captures keep the copies.
static bool captured(cudaStream_t s) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &status) == cudaSuccess) return status != cudaStreamCaptureStatusNone;
    (void)cudaGetLastError();
    return true;
}

template <bool TO_POOL>
static int swap_pages(const asynclm_shape* shape, const int32_t* page_ids, int32_t n_pages, const void* pool, void* staging,
                      void* host_image, cudaStream_t s) {
    const size_t bytes = (size_t)n_pages * page_bytes(shape);
    const int vpp = (int)(page_bytes(shape) / 16);
    const int64_t total = (int64_t)n_pages * vpp;
    const bool by_value = n_pages <= kIdsInParams && !captured(s);
    int32_t* ids_dev = reinterpret_cast<int32_t*>((char*)staging + bytes);
    IdsByValue ids;
    if (by_value) {
        std::copy(page_ids, page_ids + n_pages, ids.id);
        if (void* in_place = bytes <= kDirectBytes ? page_locked_on_device(host_image, bytes) : nullptr)
            return copy_pages<TO_POOL, true>(pool, in_place, ids, total, vpp, s);
    } else if (int rc = cuda_status(cudaMemcpyAsync(ids_dev, page_ids, (size_t)n_pages * 4, cudaMemcpyHostToDevice, s))) {
        return rc;
    }
    if (TO_POOL)
        if (int rc = cuda_status(cudaMemcpyAsync(staging, host_image, bytes, cudaMemcpyHostToDevice, s))) return rc;
    if (int rc = by_value ? copy_pages<TO_POOL, false>(pool, staging, ids, total, vpp, s)
                          : copy_pages<TO_POOL, false>(pool, staging, IdsInMemory{ids_dev}, total, vpp, s))
        return rc;
    return TO_POOL ? ASYNCLM_OK : cuda_status(cudaMemcpyAsync(host_image, staging, bytes, cudaMemcpyDeviceToHost, s));
}

}  // namespace asynclm

using namespace asynclm;

extern "C" size_t asynclm_kv_swap_staging_bytes(const asynclm_shape* shape, int32_t n_pages) {
    if (!shape || n_pages < 0) return 0;
    return (size_t)n_pages * page_bytes(shape) + (((size_t)n_pages * 4 + 255) / 256) * 256;
}

extern "C" int asynclm_kv_swap_out(const asynclm_shape* shape, const int32_t* page_ids, int32_t n_pages,
                                   const void* kv_pool, void* staging, void* host_image, void* stream) {
    if (int rc = check_swap_args(shape, page_ids, n_pages, kv_pool, staging, host_image, false)) return rc;
    if (n_pages == 0) return ASYNCLM_OK;
    return swap_pages<false>(shape, page_ids, n_pages, kv_pool, staging, host_image, (cudaStream_t)stream);
}

extern "C" int asynclm_kv_swap_in(const asynclm_shape* shape, const int32_t* page_ids, int32_t n_pages,
                                  void* kv_pool, void* staging, const void* host_image, void* stream) {
    if (int rc = check_swap_args(shape, page_ids, n_pages, kv_pool, staging, host_image, true)) return rc;
    if (n_pages == 0) return ASYNCLM_OK;
    return swap_pages<true>(shape, page_ids, n_pages, kv_pool, staging, const_cast<void*>(host_image), (cudaStream_t)stream);
}

extern "C" int asynclm_trap_decide(const asynclm_trap_model* model, int32_t context_tokens, double wait_us,
                                   int32_t* decision, double* swap_us, double* recompute_us) {
    if (!model || !decision || context_tokens < 0 || !(wait_us >= 0.0)) return ASYNCLM_ERR_INVALID_ARG;
    const double n = (double)context_tokens;
    const double s = model->swap_fixed_us + model->swap_us_per_token * n;
    const double r = model->recompute_fixed_us + model->recompute_us_per_token * n + model->recompute_us_per_token2 * n * n;
    if (swap_us) *swap_us = s;
    if (recompute_us) *recompute_us = r;
    if (s > wait_us && r > wait_us) *decision = ASYNCLM_TRAP_KEEP;
    else *decision = r < s ? ASYNCLM_TRAP_RECOMPUTE : ASYNCLM_TRAP_SWAP;
    return ASYNCLM_OK;
}
