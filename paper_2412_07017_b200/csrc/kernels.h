// Launchers of the device kernels (internal).  Each returns a cudaError_t from the launch.
#pragma once
#include <cuda_runtime.h>

#include "plan_types.h"

namespace asynclm {

// The driver's entry points are looked up once per process.
template <typename Fn>
cudaError_t driver_function(const char* name, Fn* fn) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t e = cudaGetDriverEntryPoint(name, &sym, cudaEnableDefault, &qres);
    if (e != cudaSuccess) return e;
    if (qres != cudaDriverEntryPointSuccess) return cudaErrorNotSupported;
    *fn = (Fn)sym;
    return cudaSuccess;
}

// Page-locked host memory as kernels of the current device see it, or null: pageable or managed memory, and memory that is not
// all in one allocation or one registration.
void* page_locked_on_device(const void* host, size_t bytes);

// The packed plan from page-locked host memory into the device workspace, by a kernel, for plans of these sizes.  Smaller ones belong to
// steps that the host bounds, where the question whether the workspace is page-locked costs more than the copy does; of larger ones the bus
// takes most of the time either way (none was measured: 2 MB are pages of 7 million tokens).
constexpr size_t kUploadMinBytes = 32 << 10, kUploadMaxBytes = 2 << 20;
cudaError_t upload_plan(void* dev, const void* host, size_t bytes, cudaStream_t stream);

cudaError_t launch_kv_append(const DevPlan& p, const void* k_new, const void* v_new, void* kv_pool,
                             cudaStream_t stream);

// All attention kernels of a step: span tiles and warp-body items (one fused launch when the step
// has both), writing final rows to `out` and split rows to the plan's partials.  With app.k_new set,
// only for steps without span tiles, the kernel first puts every new K/V row it is about to read into its
// page slot itself.
cudaError_t launch_attention(const DevPlan& p, const void* q, const void* kv_pool, void* out, float* lse,
                             cudaStream_t stream, AppendSrc app = AppendSrc{nullptr, nullptr, nullptr});

cudaError_t launch_lse_merge(const DevPlan& p, void* out, float* lse, cudaStream_t stream);

// Remembers `e` as the calling thread's last CUDA error (asynclm_last_cuda_error) and clears the
// runtime's sticky launch error; returns ASYNCLM_OK for cudaSuccess, else ASYNCLM_ERR_CUDA.
int cuda_status(cudaError_t e);

// ASYNCLM_OK if the current device is the one the plan was made for, else ASYNCLM_ERR_INVALID_ARG
// (ASYNCLM_ERR_CUDA if the device cannot be queried).
int check_plan_device(int plan_device);

}  // namespace asynclm
