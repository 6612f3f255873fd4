"""Which calls of a plan start early, on the CPU: csrc/api.cu built against launchers and a runtime that note what they are given.

A plan uploaded by a kernel may be read early by a launch only if another one has been accepted behind that upload: until then
every call gets the full launch, however the calls before it ended.  A capture orders nothing for launches outside of it, nor for
the next capture.
"""
import ctypes
import os
import subprocess

import pytest

from paper_2412_07017_b200 import build as lib_build

CUDA = "/usr/local/cuda/include"
PROBE = """
#include "api.cu"

static int g_refuse, g_query_fails, g_launches, g_last_error;
static unsigned long long g_capture;
static cudaError_t launched(const DevPlan& p) {
    if (g_refuse) return cudaErrorInvalidValue;
    g_launches = 10 * g_launches + 1 + (p.full_launch != 0);      // a digit for each launch: 1 early, 2 full
    return cudaSuccess;
}
namespace asynclm {
cudaError_t launch_kv_append(const DevPlan& p, const void*, const void*, void*, cudaStream_t) { return launched(p); }
cudaError_t launch_attention(const DevPlan& p, const void*, const void*, void*, float*, cudaStream_t, AppendSrc) { return launched(p); }
cudaError_t launch_lse_merge(const DevPlan&, void*, float*, cudaStream_t) { return cudaSuccess; }
}
extern "C" {
cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetLastError(void) { g_last_error = 0; return cudaSuccess; }
const char* CUDARTAPI cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t CUDARTAPI cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
#undef cudaStreamGetCaptureInfo
static cudaError_t query(cudaStreamCaptureStatus* s, unsigned long long* id) {
    if (g_query_fails) { g_last_error = 1; return cudaErrorStreamCaptureImplicit; }
    *s = g_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    if (g_capture && id) *id = g_capture - 1;
    return cudaSuccess;
}
cudaError_t CUDARTAPI cudaStreamGetCaptureInfo_v2(cudaStream_t, cudaStreamCaptureStatus* s, unsigned long long* id, cudaGraph_t*,
                                                  const cudaGraphNode_t**, size_t*) { return query(s, id); }

// capture: 0 outside of one, k > 0 inside the capture with id k - 1.  Returns the launches' digits, or -1 if the call is refused.
int call(asynclm_plan_s* plan, int which, int refuse, int capture, int query_fails) {
    g_refuse = refuse; g_capture = capture; g_query_fails = query_fails; g_launches = 0;
    void* a = (void*)256;
    int rc = which == 0 ? asynclm_kv_append(plan, a, a, a, nullptr) : which == 1 ? asynclm_attn_mixed(plan, a, a, a, nullptr, nullptr)
             : asynclm_step(plan, a, a, a, a, a, nullptr, nullptr);
    return rc ? -1 : g_launches;
}
int left_an_error(void) { return g_last_error; }
asynclm_plan_s* fresh_plan(int span_items) {
    static asynclm_plan_s plans[64];
    static int n;
    asynclm_plan_s* p = &plans[n++ % 64];
    *p = asynclm_plan_s{};
    p->magic = kPlanMagic; p->dev.total_q = 1; p->dev.num_items_tensor = span_items; p->fresh = 1;
    return p;
}
}
"""


@pytest.fixture(scope="module")
def api(tmp_path_factory):
    if not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no CUDA headers here")
    d = tmp_path_factory.mktemp("api")
    src, lib = os.path.join(d, "probe.cpp"), os.path.join(d, "probe.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CUDA, "-I", lib_build.CSRC, "-I", lib_build.INCLUDE, "-o", lib, src], check=True)
    p = ctypes.CDLL(lib)
    p.fresh_plan.restype = ctypes.c_void_p
    p.call.argtypes = [ctypes.c_void_p] + [ctypes.c_int] * 4
    return p


APPEND, ATTENTION, STEP = range(3)


@pytest.mark.parametrize("first", [APPEND, ATTENTION, STEP])
@pytest.mark.parametrize("second", [APPEND, ATTENTION, STEP])
@pytest.mark.parametrize("span_items", [0, 1])
def test_the_first_launch_that_is_accepted_is_a_full_one(api, first, second, span_items):
    digits = lambda which, full: 10 * (1 + full) + 1 if which == STEP and span_items else 1 + full
    plan = api.fresh_plan(span_items)
    assert api.call(plan, first, 1, 0, 0) == -1
    assert api.call(plan, first, 1, 0, 0) == -1      # a retry that is refused, too
    assert api.call(plan, second, 0, 0, 0) == digits(second, True)
    assert api.call(plan, first, 0, 0, 0) == digits(first, False)


@pytest.mark.parametrize("which", [APPEND, ATTENTION, STEP])
def test_each_capture_and_what_is_outside_have_a_first_launch(api, which):
    plan = api.fresh_plan(0)
    for capture in (1, 2):      # (the first with id 0)
        assert api.call(plan, which, 1, capture, 0) == -1
        assert api.call(plan, which, 0, capture, 0) == 2
        assert api.call(plan, which, 0, capture, 0) == 1
    assert api.call(plan, which, 0, 0, 0) == 2
    assert api.call(plan, which, 0, 0, 0) == 1
    assert api.call(plan, which, 0, 3, 0) == 1


@pytest.mark.parametrize("which", [APPEND, ATTENTION, STEP])
def test_a_stream_whose_capture_state_is_unknown_orders_nothing(api, which):
    plan = api.fresh_plan(0)
    assert api.call(plan, which, 0, 0, 1) == 2
    assert not api.left_an_error()
    assert api.call(plan, which, 0, 0, 0) == 2
    assert api.call(plan, which, 0, 0, 0) == 1


def test_every_launch_of_a_plan_goes_through_the_same_rule():
    """The entry points with device code beside them, by their text: what they launch first is reported to PlanUse."""
    for name, n in (("api.cu", 4), ("attn_static_scratch.cu", 1), ("kv_append_rope.cu", 1)):
        with open(os.path.join(lib_build.CSRC, name)) as f:
            assert f.read().count("use.launched(launch_") == n, name
