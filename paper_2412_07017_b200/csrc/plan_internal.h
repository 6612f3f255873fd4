// Host-side plan object and planner constants (internal).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "asynclm.h"
#include "plan_types.h"

namespace asynclm {

constexpr uint64_t kPlanMagic = 0x4153594e434c4d31ull;   // "ASYNCLM1"

// Persistent CTAs per SM of the kernel that runs the warp body.
constexpr int kCudaSlotsPerSm = 1;
// Fixed cost of starting an item, in units of one 128-token KV tile, used when balancing CTAs.
constexpr int kCudaItemOverheadTiles = 1;
constexpr int kTensorItemOverheadTiles = 4;   // an item boundary costs the span body 2 to 4 tiles

int tensor_tile_tokens(int group);

}  // namespace asynclm

struct asynclm_plan_s {
    uint64_t magic;
    asynclm_shape shape;
    asynclm_plan_info info;
    asynclm::DevPlan dev;
    const asynclm::Unit* h_units;
    const asynclm::Item* h_items;
    const int32_t* h_item_cta;
    const int32_t* h_kv_len_before;
    int32_t h_units_path_split;   // items [0, this) are warp-body items, the rest span items
    int32_t device;
    int32_t host_only;
    int32_t max_q_len;            // longest span of the step
    mutable int32_t fresh;        // the upload was a kernel, and no launch has been ordered behind it yet (see PlanUse)
    mutable unsigned long long captured_in;      // 1 + the id of the last stream capture that a launch of a fresh plan went into, or 0
};

namespace asynclm {

// The device plan for one call.  The kernels read the plan ahead of their wait for the kernel in front, which may only be as far as its
// trigger then: what a copy in the stream wrote is complete and in no cache by that time, what a kernel in front is
// writing need not be.  So the first launch behind an upload by kernel starts when that has completed, as behind a copy, and the others, which
// come behind that one, early again.  A launch counts as the first when it has been accepted: behind a refused call the next one is
// the first again.  (A captured launch orders nothing now: each capture has a first launch of its own, and the plan
// stays fresh for launches outside.  So does a launch whose stream does not say whether it is being captured.)
class PlanUse {
    const asynclm_plan_s* plan;
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusInvalidated;
    unsigned long long id = 0;

  public:
    DevPlan dev;

    PlanUse(const asynclm_plan_s* p, cudaStream_t stream) : plan(p), dev(p->dev) {
        dev.full_launch = 0;
        if (__atomic_load_n(&plan->fresh, __ATOMIC_ACQUIRE) == 0) return;
        if (cudaStreamGetCaptureInfo(stream, &status, &id) != cudaSuccess) {
            (void)cudaGetLastError();
            status = cudaStreamCaptureStatusInvalidated;
        }
        dev.full_launch = status != cudaStreamCaptureStatusActive || __atomic_load_n(&plan->captured_in, __ATOMIC_ACQUIRE) != id + 1;
    }

    // Takes and returns the outcome of the call's first launch with `dev`; what the call launches behind it starts early.
    cudaError_t launched(cudaError_t e) {
        if (e != cudaSuccess || dev.full_launch == 0) return e;
        if (status == cudaStreamCaptureStatusActive) __atomic_store_n(&plan->captured_in, id + 1, __ATOMIC_RELEASE);
        if (status == cudaStreamCaptureStatusNone) __atomic_store_n(&plan->fresh, 0, __ATOMIC_RELEASE);
        dev.full_launch = 0;
        return e;
    }
};

}  // namespace asynclm
