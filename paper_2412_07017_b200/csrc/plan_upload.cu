// A plan's way to the GPU as a kernel that reads it out of page-locked host memory.
//
// A copy in the stream stands between two steps' kernels for 12-17 us, whatever its 100-300 KB take on the bus: the copy engine
// starts when the kernel in front has been flushed, and the kernel behind when the copy has.  This kernel is resident
// while the kernel in front runs out, has requested its share from the host by then and only stores it behind the wait.
// (Whole passes, copy | kernel: four steps of 256 sequences, planned anew each, 816 | 777 us; 64 decoding sequences in 8 layers 669 |
// 660, 24 spans in 4 layers 344 | 337, 4 decoding sequences in 32 layers 386 | 377, 32 of head_dim 64 in 16 layers 781 | 771.)
#include <cuda.h>

#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace asynclm {

namespace {

constexpr int kUploadCtas = 148, kUploadThreads = 256, kUploadAhead = 4;      // 16-byte vectors of a thread, at most, all requested ahead of the wait
// Shared memory that holds an SM to five of these CTAs; nothing is kept in it.  They start where the kernel in front has left first, and
// what piles up there reads the bus more slowly (four steps of 256 sequences with eight CTAs an SM 797 us, with five 790, with one or two the same).
constexpr size_t kUploadSpread = 40 << 10;
static_assert(kUploadMaxBytes <= (size_t)16 * kUploadCtas * kUploadThreads * kUploadAhead, "the largest plan is read in one pass");

__global__ void __launch_bounds__(kUploadThreads)
plan_upload_kernel(uint4* __restrict__ dev, const uint4* host, int n) {
    const int step = gridDim.x * kUploadThreads;
    const int i = blockIdx.x * kUploadThreads + threadIdx.x;
    uint4 v[kUploadAhead];
#pragma unroll
    for (int k = 0; k < kUploadAhead; ++k)
        if (i + k * step < n) v[k] = ld_host_v4(host + i + k * step);
    pdl_wait();      // the workspace belongs to the kernels in front until those have completed
#pragma unroll
    for (int k = 0; k < kUploadAhead; ++k)
        if (i + k * step < n) dev[i + k * step] = v[k];
    // No early trigger: the kernels behind read the plan ahead of their own wait (see PlanUse).
}

typedef CUresult (*PointerAttributesFn)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);

}  // namespace

void* page_locked_on_device(const void* host, size_t bytes) {
    static std::atomic<PointerAttributesFn> attributes_fn{nullptr};
    PointerAttributesFn attributes = attributes_fn.load(std::memory_order_acquire);
    if (attributes == nullptr) {
        if (driver_function("cuPointerGetAttributes", &attributes) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        attributes_fn.store(attributes, std::memory_order_release);
    }
    unsigned type = 0, managed = 0;
    CUdeviceptr dev = 0, start = 0;
    size_t size = 0;
    CUpointer_attribute which[5] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_IS_MANAGED, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                    CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* to[5] = {&type, &managed, &dev, &start, &size};
    if (attributes(5, which, to, (CUdeviceptr)(uintptr_t)host) != CUDA_SUCCESS) return nullptr;
    if (type != CU_MEMORYTYPE_HOST || managed != 0 || dev == 0 || dev < start || dev - start > size || size - (dev - start) < bytes) return nullptr;
    return (void*)(uintptr_t)dev;
}

cudaError_t upload_plan(void* dev, const void* host, size_t bytes, cudaStream_t stream) {
    if (bytes > kUploadMaxBytes) return cudaErrorInvalidValue;
    const int n = (int)(bytes / 16);      // (the sections of a plan are multiples of 256 bytes)
    const int blocks = std::min(kUploadCtas, (n + kUploadThreads - 1) / kUploadThreads);
    return launch_pdl(plan_upload_kernel, dim3(blocks), dim3(kUploadThreads), kUploadSpread, stream, (uint4*)dev, (const uint4*)host, n);
}

}  // namespace asynclm
