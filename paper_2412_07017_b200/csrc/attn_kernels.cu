// The attention kernels' entry points and launchers.
//
// Three kernels are built from two bodies (attn_append_tc.cuh: span tiles on tcgen05, attn_decode.cuh: decode
// rows and short spans on warp-level MMAs):
//   attn_fused_kernel      a persistent CTA first runs its span items, then takes warp-body items
//                          (a CTA without span tiles skips the tensor-memory set-up altogether).
//                          One launch instead of two: the fixed cost of a launch (about 10 us of
//                          start-up and tail per kernel at 148 CTAs) is paid once, and a CTA that is
//                          done with its span tiles early moves on to decode rows at once.
//   attn_append_tc_kernel  steps that have span tiles only
//   attn_decode_kernel     steps without span tiles
// All are launched with programmatic stream serialization and wait for the kernel in front of them
// (normally the KV append) right before they first touch the pool.
#include <algorithm>
#include <atomic>

#include "attn_append_tc.cuh"
#include "attn_decode.cuh"

namespace asynclm {

namespace {

constexpr int kMaxSmem = 232448;

__device__ __forceinline__ uint8_t* aligned_smem(uint8_t* raw) {
    return (uint8_t*)(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
}

template <int D, int G, bool APPEND>
__global__ void __launch_bounds__(dec::kThreads, 1)
attn_decode_kernel(DevPlan p, const __grid_constant__ CUtensorMap kv_map, const __nv_bfloat16* pool, const __nv_bfloat16* __restrict__ q,
                   __nv_bfloat16* __restrict__ out, float* __restrict__ lse, int S, AppendSrc app) {
    extern __shared__ uint8_t smem_raw[];
    pdl_trigger();      // the split-KV merge behind this kernel may start its prologue
    if (threadIdx.x == 0) { trace_mark(0); trace_set(1, 0); trace_set(5, 0); trace_set(6, 0); trace_set(7, 0); }
    dec::decode_body<D, G, APPEND, true>(p, &kv_map, pool, q, out, lse, S, aligned_smem(smem_raw), app);
}

template <int D, int G>
__global__ void __launch_bounds__(tc::kThreads, 1)
attn_append_tc_kernel(DevPlan p, const __grid_constant__ CUtensorMap span_map, const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* pool,
                      __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
    extern __shared__ uint8_t smem_raw[];
    pdl_trigger();      // the kernel behind this one may start its prologue; it waits for this grid to complete
    if (threadIdx.x == 0) {
        trace_mark(0);
        for (int s = 8; s < 16; ++s) trace_set(s, 0);
    }
    tc::tc_body<D, G, true>(p, &span_map, q, pool, out, lse, aligned_smem(smem_raw));
    if (threadIdx.x == 0) trace_mark(1);
}

template <int D, int G>
__global__ void __launch_bounds__(tc::kThreads, 1)
attn_fused_kernel(DevPlan p, const __grid_constant__ CUtensorMap kv_map, const __grid_constant__ CUtensorMap span_map,
                  const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* pool, __nv_bfloat16* __restrict__ out, float* __restrict__ lse,
                  int S) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = aligned_smem(smem_raw);
    pdl_trigger();      // the split-KV merge behind this kernel may start its prologue
    if (threadIdx.x == 0) { trace_mark(0); trace_set(1, 0); trace_set(5, 0); trace_set(6, 0); trace_set(7, 0); }
    const int32_t* head = p.cta_heads + (size_t)blockIdx.x * kHeadWords;
    // bring the whole header and the tensor map close now: the decode phase of a CTA that starts with
    // span tiles finds them in L2 when it gets there
    if (threadIdx.x < 3) asm volatile("prefetch.global.L2 [%0];" ::"l"(head + 32 * threadIdx.x));
    if (threadIdx.x == 32) asm volatile("prefetch.tensormap [%0];" ::"l"(&kv_map));
    if (head[0] == head[1]) {
        // no span tiles for this CTA: straight to its decode rows, without the tensor-memory set-up
        dec::decode_body<D, G, false, false>(p, &kv_map, nullptr, q, out, lse, S, smem, AppendSrc{});
        return;
    }
    if (threadIdx.x == 0) {
        for (int s = 8; s < 16; ++s) trace_set(s, 0);
    }
    tc::tc_body<D, G, false>(p, &span_map, q, pool, out, lse, smem);
    if (threadIdx.x == 0) trace_mark(1);
    if (head[2] == head[3] && p.queue_count == 0) return;      // nothing left for the warp body
    __syncthreads();      // tensor memory released, shared memory free for the second phase
    dec::decode_body<D, G, false, false>(p, &kv_map, nullptr, q, out, lse, S, smem, AppendSrc{});
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

typedef CUresult (*ReplaceAddressFn)(CUtensorMap*, void*);

// The pool as the two bodies read it, landed with the 128-byte swizzle:
//   kv    (64 values, 16 slots, d / 64 row halves, Hkv, pages x K|V), a box is one page's K and V blocks of one kv head
//         (dec::tma_page_kv)
//   span  (64 values, 8 slots, d / 64 row halves, 2 groups of 8 slots, pages x K|V x Hkv), a box is one block (tc::tma_page)
enum PoolMap { kKvMap, kSpanMap };

constexpr int64_t kMaxMapPages = 0x3fffffff;

cudaError_t make_pool_map(PoolMap kind, const DevPlan& p, const void* pool, CUtensorMap* map) {
    static std::atomic<EncodeTiledFn> encode_fn{nullptr};
    EncodeTiledFn encode = encode_fn.load(std::memory_order_acquire);
    if (encode == nullptr) {
        cudaError_t e = driver_function("cuTensorMapEncodeTiled", &encode);
        if (e != cudaSuccess) return e;
        encode_fn.store(encode, std::memory_order_release);
    }
    const cuuint64_t d = (cuuint64_t)p.head_dim, hkv = (cuuint64_t)p.num_kv_heads;
    if (p.num_pages <= 0) return cudaErrorInvalidValue;
    // (the pages that a tensor map can count hold more than any device's memory)
    const cuuint64_t blocks = 2 * (cuuint64_t)std::min(p.num_pages, kMaxMapPages);
    const cuuint64_t dims_kv[5] = {64, kPage, d / 64, hkv, blocks}, strides_kv[4] = {d * 2, 128, kPage * d * 2, hkv * kPage * d * 2};
    const cuuint64_t dims_span[5] = {64, 8, d / 64, 2, std::min<cuuint64_t>(blocks * hkv, INT32_MAX)};
    const cuuint64_t strides_span[4] = {d * 2, 128, 8 * d * 2, kPage * d * 2};
    const cuuint32_t box_kv[5] = {64, kPage, (cuuint32_t)(d / 64), 1, 2}, box_span[5] = {64, 8, (cuuint32_t)(d / 64), 2, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(pool), kind == kKvMap ? dims_kv : dims_span,
                              kind == kKvMap ? strides_kv : strides_span, kind == kKvMap ? box_kv : box_span, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per kernel and device instead of once per launch.
// The kernel is a template VALUE: kernels of one signature share a pointer type, and a flag per type
// would let the first of them stand for all.
template <auto kernel>
cudaError_t allow_smem(size_t bytes) {
    static std::atomic<unsigned long long> done{0};      // one per kernel instantiation; bit = device (first 64)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (bit != 0 && (done.load(std::memory_order_acquire) & bit) != 0) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && bit != 0) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// A pool's tensor map: that of its shape, of which the last few are kept per thread and kind, with its address put in.
// (The layers of a model have a pool each; encoding a launch's map anew takes longer than the address.)
cudaError_t pool_map(PoolMap kind, const DevPlan& p, const void* pool, CUtensorMap* map) {
    struct Entry { int64_t pages; int hkv, d; CUtensorMap map; };
    constexpr int kEntries = 8;
    thread_local Entry cache[2][kEntries] = {};
    thread_local int next[2] = {};
    static std::atomic<ReplaceAddressFn> replace_fn{nullptr};
    ReplaceAddressFn replace = replace_fn.load(std::memory_order_acquire);
    if (replace == nullptr) {
        cudaError_t e = driver_function("cuTensorMapReplaceAddress", &replace);
        if (e != cudaSuccess) return e;
        replace_fn.store(replace, std::memory_order_release);
    }
    for (const Entry& x : cache[kind])
        if (x.pages == p.num_pages && x.hkv == p.num_kv_heads && x.d == p.head_dim) {
            *map = x.map;
            return replace(map, const_cast<void*>(pool)) == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
        }
    const cudaError_t e = make_pool_map(kind, p, pool, map);
    if (e == cudaSuccess) {
        cache[kind][next[kind]] = Entry{p.num_pages, p.num_kv_heads, p.head_dim, *map};
        next[kind] = (next[kind] + 1) % kEntries;
    }
    return e;
}

template <int D>
constexpr int decode_stages() {
    int S = dec::kMaxStages;
    while (S > 2 && dec::smem_bytes<D>(S) > (size_t)kMaxSmem) --S;
    return S;
}

template <int D, int G, bool APPEND>
cudaError_t launch_decode(const DevPlan& p, const void* q, const void* pool, void* out, float* lse,
                          cudaStream_t stream, AppendSrc app) {
    const int S = decode_stages<D>();
    const size_t smem = dec::smem_bytes<D>(S);
    cudaError_t e = allow_smem<attn_decode_kernel<D, G, APPEND>>(smem);
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    if (p.num_pages > kMaxMapPages) return cudaErrorInvalidValue;
    e = pool_map(kKvMap, p, pool, &map);
    if (e != cudaSuccess) return e;
    return launch_when(!p.full_launch, attn_decode_kernel<D, G, APPEND>, dim3(p.num_ctas_cuda), dim3(dec::kThreads), smem, stream, p, map,
                      (const __nv_bfloat16*)pool, (const __nv_bfloat16*)q, (__nv_bfloat16*)out, lse, S, app);
}

template <int D, int G>
cudaError_t launch_tensor(const DevPlan& p, const void* q, const void* pool, void* out, float* lse, cudaStream_t stream) {
    constexpr size_t smem = tc::Geometry<D>::SMEM_BYTES;
    cudaError_t e = allow_smem<attn_append_tc_kernel<D, G>>(smem);
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    e = pool_map(kSpanMap, p, pool, &map);
    if (e != cudaSuccess) return e;
    return launch_when(!p.full_launch, attn_append_tc_kernel<D, G>, dim3(p.num_ctas_tensor), dim3(tc::kThreads), smem, stream,
                      p, map, (const __nv_bfloat16*)q, (const __nv_bfloat16*)pool, (__nv_bfloat16*)out, lse);
}

template <int D, int G>
cudaError_t launch_fused(const DevPlan& p, const void* q, const void* pool, void* out, float* lse, cudaStream_t stream) {
    constexpr int S = decode_stages<D>();
    constexpr size_t smem = std::max<size_t>(dec::smem_bytes<D>(S), tc::Geometry<D>::SMEM_BYTES);
    static_assert(dec::smem_bytes<D>(S) - 1024 <= tc::Geometry<D>::OFF_BAR, "the span body's barriers stay clear of the warp body");
    cudaError_t e = allow_smem<attn_fused_kernel<D, G>>(smem);
    if (e != cudaSuccess) return e;
    CUtensorMap kv_map, span_map;
    if (p.num_pages > kMaxMapPages) return cudaErrorInvalidValue;
    e = pool_map(kKvMap, p, pool, &kv_map);
    if (e == cudaSuccess) e = pool_map(kSpanMap, p, pool, &span_map);
    if (e != cudaSuccess) return e;
    return launch_when(!p.full_launch, attn_fused_kernel<D, G>, dim3(p.num_ctas_cuda), dim3(tc::kThreads), smem, stream, p, kv_map, span_map,
                      (const __nv_bfloat16*)q, (const __nv_bfloat16*)pool, (__nv_bfloat16*)out, lse, S);
}

template <int D, int G>
cudaError_t launch_attention_impl(const DevPlan& p, const void* q, const void* kv_pool, void* out, float* lse,
                                  cudaStream_t stream, AppendSrc app) {
    const bool has_tensor = p.num_items_tensor > 0, has_cuda = p.num_items_cuda > 0;
    if (app.k_new != nullptr)      // the warp body only
        return has_tensor || !has_cuda ? cudaErrorInvalidValue : launch_decode<D, G, true>(p, q, kv_pool, out, lse, stream, app);
    if (has_tensor && has_cuda && p.num_ctas_tensor == p.num_ctas_cuda)
        return launch_fused<D, G>(p, q, kv_pool, out, lse, stream);
    if (has_tensor)
        if (cudaError_t e = launch_tensor<D, G>(p, q, kv_pool, out, lse, stream)) return e;
    // a decode kernel behind a tensor kernel would have to wait for it to finish (pdl_wait), which is what
    // stream order gives anyway
    return has_cuda ? launch_decode<D, G, false>(p, q, kv_pool, out, lse, stream, app) : cudaSuccess;
}

template <int D>
cudaError_t launch_attention_d(const DevPlan& p, const void* q, const void* kv_pool, void* out, float* lse,
                               cudaStream_t stream, AppendSrc app) {
    switch (p.group) {
        case 1: return launch_attention_impl<D, 1>(p, q, kv_pool, out, lse, stream, app);
        case 2: return launch_attention_impl<D, 2>(p, q, kv_pool, out, lse, stream, app);
        case 4: return launch_attention_impl<D, 4>(p, q, kv_pool, out, lse, stream, app);
        case 8: return launch_attention_impl<D, 8>(p, q, kv_pool, out, lse, stream, app);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_attention(const DevPlan& p, const void* q, const void* kv_pool, void* out, float* lse,
                             cudaStream_t stream, AppendSrc app) {
    if (p.head_dim == 128) return launch_attention_d<128>(p, q, kv_pool, out, lse, stream, app);
    if (p.head_dim == 64) return launch_attention_d<64>(p, q, kv_pool, out, lse, stream, app);
    return cudaErrorInvalidValue;
}

}  // namespace asynclm

#ifdef ASYNCLM_TRACE
// Debug builds only: copies the per-CTA time stamps of the last attention launch to the host
// (synchronises the device).  out: [1024][8] unsigned 64-bit.
extern "C" int asynclm_trace_read(unsigned long long* out) {
    return cudaMemcpyFromSymbol(out, asynclm::g_trace, sizeof(asynclm::g_trace)) == cudaSuccess ? 0 : -5;
}
// The event log of the first CTAs: out [4][11][512] unsigned 64-bit (cycle << 8 | event); clears it.
extern "C" int asynclm_trace_events_read(unsigned long long* out) {
    if (cudaMemcpyFromSymbol(out, asynclm::g_events, sizeof(asynclm::g_events)) != cudaSuccess) return -5;
    void* dev = nullptr;
    if (cudaGetSymbolAddress(&dev, asynclm::g_events) != cudaSuccess) return -5;
    return cudaMemset(dev, 0, sizeof(asynclm::g_events)) == cudaSuccess ? 0 : -5;
}
#endif