// Interrupt append with the rotary position embedding fused in: the form the append takes in a
// multi-layer model of the Llama family (the models the paper serves, Section 6), where a key is
// rotated by its position before it is cached.  New token i of sequence b sits at position ctx_b + i
// (Section 3.2: the block goes to the end of the context).  K rows are rotated ("rotate-half" pairs
// (j, j + d/2), angle pos * theta^(-2j/d)) and written to their page slots, V rows are copied bit for
// bit, and, if asked, the step's query rows are rotated in place by the same positions.
//
// Angles and the rotation are evaluated in fp64 and rounded once (fp64 -> fp32 -> bf16, nearest even):
// positions reach 10^5, where an fp32 angle would already be off by several thousandths of a radian.
// An fp64 sincos and exp2 cost a few hundred instructions, and an angle depends on the token and the
// pair only, so a CTA takes whole tokens: their d / 2 angles are evaluated once, a thread each, kept in
// shared memory and used by all heads.  (One thread per (head, 8 pairs) that evaluated its own eight
// angles, one after the other, was bound by that arithmetic: 10.1 us against 6.2 so for 314 tokens of
// 32 + 8 heads, d = 128, and 142 us against 41 for 8192 tokens, whose rows take 31 us at the copy rate.)
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include "asynclm.h"
#include "common.cuh"
#include "kernels.h"
#include "plan_internal.h"
#include "rope_grid.h"

namespace asynclm {

namespace {

__device__ __forceinline__ float bf16_to_f32(unsigned short b) { return __uint_as_float((unsigned)b << 16); }
__device__ __forceinline__ unsigned short f64_to_bf16(double x) {
    const __nv_bfloat16 h = __float2bfloat16_rn(__double2float_rn(x));
    return *reinterpret_cast<const unsigned short*>(&h);
}

// One row of one head as a thread holds it: 16-byte vectors v and v + half_vecs (values 8v .. 8v+7 and
// their partners d/2 further), and those of the V row beside a K row.
struct RopeRow { uint4 lo, hi, vlo, vhi; };

// Grid: one CTA per `tokens` (<= kRopeTokens) new tokens.  A thread rotates its part of a row and goes on
// to a later (token, head) with the same v, whose loads it has requested before.  Heads: K rows
// [T][Hkv][d] first (written to the pool, the V row beside them copied) and then, optionally, Q rows
// [T][Hq][d] (rewritten in place).
__global__ void __launch_bounds__(kRopeThreads)
kv_append_rope_kernel(DevPlan p, const uint4* __restrict__ k_new, const uint4* __restrict__ v_new,
                      uint4* __restrict__ pool, uint4* __restrict__ q, double log2_theta, int tokens) {
    // (cos, sin) of pair 8 v + k of token i at [i][k][v]: the threads of a warp read consecutive entries
    extern __shared__ double2 rot[];      // [tokens][64]
    int64_t* slot = reinterpret_cast<int64_t*>(rot + tokens * 64);
    pdl_trigger();   // the attention kernel may start its prologue; it waits for this grid before reading the pool
    const int d = p.head_dim, half_vecs = d / 16;                 // vectors in half a row: 8 or 4
    const int heads_k = p.num_kv_heads, heads_q = q != nullptr ? p.num_q_heads : 0, heads = heads_k + heads_q;
    const int v = threadIdx.x % half_vecs, step = blockDim.x / half_vecs;
    const int r0 = blockIdx.x * tokens, n = min(tokens, p.total_q - r0);
    auto load = [&](int i, int h) {
        RopeRow x{};
        if (i >= n) return x;
        if (h < heads_k) {
            const size_t at = ((size_t)(r0 + i) * heads_k + h) * (2 * half_vecs) + v;
            x.lo = k_new[at]; x.hi = k_new[at + half_vecs];
            x.vlo = v_new[at]; x.vhi = v_new[at + half_vecs];
        } else {
            const size_t at = ((size_t)(r0 + i) * heads_q + (h - heads_k)) * (2 * half_vecs) + v;
            x.lo = q[at]; x.hi = q[at + half_vecs];
        }
        return x;
    };
    auto advance = [&](int& i, int& h) {
        for (h += step; h >= heads && i < n; h -= heads) ++i;
    };
    int i = 0, h = threadIdx.x / half_vecs;
    for (; h >= heads && i < n; h -= heads) ++i;
    // The rows and the pool belong to the kernels in front until those have completed; the angles come from the plan.  Where
    // about all CTAs start at once, the angles overlap the tail of the kernel in front, and the rows are requested behind
    // the wait that follows.  In a longer grid most CTAs start when that kernel has completed: they request their rows first.
    // (us a launch, call after call, rows first | angles first: 320 tokens of 32/8 heads 4.9 | 4.3, 512 7.3 | 6.5, 2048 16.0 |
    // 16.0, 2400 16.7 | 17.7, 3000 19.1 | 18.4, 4096 24.6 | 25.3, 8192 43.0 | 44.4, with at most four tokens to a CTA.)
    const bool angles_first = gridDim.x <= (unsigned)kRopeFirstCtas;
    RopeRow cur{};
    if (!angles_first) {
        pdl_wait();
        cur = load(i, h);
    }
    for (int a = threadIdx.x; a < n * (d / 2); a += blockDim.x) {
        const int ti = a / (d / 2), j = a % (d / 2), r = r0 + ti;
        const int b = __ldg(p.row_seq + r);
        const int pos = __ldg(p.kv_len_before + b) + r - __ldg(p.q_indptr + b);
        double s, c;
        sincos((double)pos * exp2(-2.0 * (double)j / (double)d * log2_theta), &s, &c);
        rot[ti * 64 + (j % 8) * half_vecs + j / 8] = make_double2(c, s);
        if (j == 0) {
            const int64_t ps = __ldg(p.row_slot + r);
            slot[ti] = page_ok(ps / kPage, p.num_pages, p.status, kStatusBadPageAppend) ? ps : -1;
        }
    }
    if (angles_first) {
        pdl_wait();
        cur = load(i, h);
    }
    __syncthreads();
    while (i < n) {
        int ni = i, nh = h;
        advance(ni, nh);
        const RopeRow next = load(ni, nh);
        const unsigned short* xl = reinterpret_cast<const unsigned short*>(&cur.lo);
        const unsigned short* xh = reinterpret_cast<const unsigned short*>(&cur.hi);
        uint4 olo, ohi;
        unsigned short* yl = reinterpret_cast<unsigned short*>(&olo);
        unsigned short* yh = reinterpret_cast<unsigned short*>(&ohi);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const double2 cs = rot[i * 64 + k * half_vecs + v];
            const double a = (double)bf16_to_f32(xl[k]), bb = (double)bf16_to_f32(xh[k]);
            yl[k] = f64_to_bf16(a * cs.x - bb * cs.y);
            yh[k] = f64_to_bf16(bb * cs.x + a * cs.y);
        }
        if (h < heads_k) {
            const int64_t ps = slot[i];
            if (ps >= 0) {      // (the checked build leaves a bad page out)
                const size_t kd = pool_row_offset(ps / kPage, 0, h, (int)(ps % kPage), heads_k, d) / 8 + v;
                pool[kd] = olo;
                pool[kd + half_vecs] = ohi;
                // the V row of the same (token, head): a bit copy
                const size_t vd = pool_row_offset(ps / kPage, 1, h, (int)(ps % kPage), heads_k, d) / 8 + v;
                pool[vd] = cur.vlo;
                pool[vd + half_vecs] = cur.vhi;
            }
        } else {
            const size_t at = ((size_t)(r0 + i) * heads_q + (h - heads_k)) * (2 * half_vecs) + v;
            q[at] = olo;
            q[at + half_vecs] = ohi;
        }
        cur = next;
        i = ni;
        h = nh;
    }
}

}  // namespace

}  // namespace asynclm

extern "C" int asynclm_kv_append_rope(const asynclm_plan_t* plan, const void* k_new, const void* v_new, void* kv_pool,
                                      void* q_inout, double rope_theta, void* stream) {
    using namespace asynclm;
    if (!plan || plan->magic != kPlanMagic || plan->host_only || !(rope_theta > 1.0)) return ASYNCLM_ERR_INVALID_ARG;
    if (plan->dev.total_q == 0) return ASYNCLM_OK;
    if (!k_new || !v_new || !kv_pool || (((uintptr_t)k_new | (uintptr_t)v_new | (uintptr_t)kv_pool | (uintptr_t)q_inout) & 15) != 0)
        return ASYNCLM_ERR_INVALID_ARG;
    if (int rc = check_plan_device(plan->device)) return rc;
    PlanUse use(plan, (cudaStream_t)stream);
    const DevPlan& p = use.dev;
    const int heads = p.num_kv_heads + (q_inout ? p.num_q_heads : 0);
    const int tokens = rope_tokens(p.total_q, heads, p.head_dim), threads = rope_threads(tokens, heads, p.head_dim);
    return cuda_status(use.launched(launch_when(!p.full_launch, kv_append_rope_kernel, dim3((p.total_q + tokens - 1) / tokens), dim3(threads), rope_smem(tokens),
                                                (cudaStream_t)stream, p, (const uint4*)k_new, (const uint4*)v_new, (uint4*)kv_pool,
                                                (uint4*)q_inout, log2(rope_theta), tokens)));
}
