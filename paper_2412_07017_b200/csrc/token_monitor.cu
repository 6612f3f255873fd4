// Token monitor's hook into next-token selection (paper Section 5.1): a finite-state machine over CML
// (Section 3) decides which tokens a sequence may produce next, [INTR] is never among them (interrupts
// are injected by the system, not generated), the allowed token with the largest logit is taken
// (lowest id among equals; NaN never), and the state machine reports a finished function call, a
// finished trap and whether the sequence is inside a function-call block (the critical section in
// which interrupts are deferred, Section 3.2).
//
// The logits are streamed once (16-byte loads, several CTAs per sequence): the kernel is bound by HBM,
// vocab * element size bytes per sequence.  The mask costs nothing per element: the scan leaves the five
// CML tokens out, which only the few vectors that hold one have to look at, and the CML tokens that the
// state allows, two at most, are fetched by their ids and compete at the end.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "asynclm.h"
#include "common.cuh"
#include "kernels.h"

namespace asynclm {

namespace {

constexpr int kMonThreads = 256;
constexpr int kMonVecs = 8;                        // 16-byte vectors in flight per thread
enum { kText = 0, kCall = 1, kBody = 2, kTrap = 3 };

struct Best {
    float v;
    int i;
};
__device__ __forceinline__ bool better(float v, int i, const Best& b) { return v > b.v || (v == b.v && i < b.i); }

__device__ __forceinline__ bool is_special(int i, const asynclm_cml_tokens& t) {
    return i == t.call || i == t.intr || i == t.trap || i == t.end || i == t.head;
}

template <typename T> __device__ __forceinline__ float to_f32(T x);
template <> __device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

// (value, id) as one 64-bit key whose unsigned order is "larger value first, then lower id": floats map
// to unsigned integers monotonically (sign bit flipped for positives, all bits for negatives), the id
// goes in complemented.  Key 0 means "nothing yet" (no real candidate maps to it: -NaN patterns never
// enter, and -inf maps to 0x007fffff in the upper half).
__device__ __forceinline__ unsigned long long pack_key(float v, int i) {
    const unsigned u = __float_as_uint(v + 0.f);      // -0 becomes +0: the two are equal, so the lower id wins
    const unsigned ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)ord << 32) | (unsigned)(0x7fffffff - i);
}
constexpr unsigned long long kNoCandidate = 1ull;      // below every candidate's key, too
__device__ __forceinline__ Best unpack_key(unsigned long long k) {
    if (k <= kNoCandidate) return Best{-INFINITY, INT_MAX};
    const unsigned ord = (unsigned)(k >> 32);
    const unsigned u = (ord & 0x80000000u) ? (ord & 0x7fffffffu) : ~ord;
    return Best{__uint_as_float(u), 0x7fffffff - (int)(unsigned)(k & 0xffffffffu)};
}

template <typename T> struct Vec;
template <> struct Vec<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ unsigned max2(unsigned a, unsigned b) {
        unsigned r;
        asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
        return r;
    }
    // largest of the 8 values of a 16-byte vector (NaN drops out of max)
    static __device__ __forceinline__ float vmax(const uint4& w) {
        const unsigned m = max2(max2(w.x, w.y), max2(w.z, w.w));
        return fmaxf(fmaxf(bf16_lo(m), bf16_hi(m)), -INFINITY);      // (-inf where all are NaN)
    }
    static __device__ __forceinline__ float at(const uint4& w, int k) {
        const unsigned u[4] = {w.x, w.y, w.z, w.w};
        return (k & 1) ? bf16_hi(u[k >> 1]) : bf16_lo(u[k >> 1]);
    }
};
template <> struct Vec<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ float vmax(const uint4& w) {
        return fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)), fmaxf(__uint_as_float(w.z), __uint_as_float(w.w)));
    }
    static __device__ __forceinline__ float at(const uint4& w, int k) {
        const unsigned u[4] = {w.x, w.y, w.z, w.w};
        return __uint_as_float(u[k]);
    }
};

// Largest ordinary element (no CML token) of vectors [j_begin, j_end) of a row (stride of the CTA's
// threads), lowest id among equals.  Per vector only its maximum is computed; the position inside the
// best vector is found at the end in the thread's copy of that one vector.  Only the vectors that hold a CML token
// have their elements looked at: when all vectors of a stretch with one were, the CTA that had it finished
// last (15.8 us a call instead of 20.5 for 256 bf16 rows of 128 256).
// The first vectors are requested before the row's state is known, and the best vector stays in registers instead of being
// read again at the end, because both stood as a round trip to memory of their own in every CTA (us a call from a graph,
// before | now, with the two slices' trade below: bf16 rows of 128 256, 256 | 148 | 64 | 8 | 1 of them: 14.1 | 10.7 | 8.3 | 5.3 | 4.7
// before, 12.7 | 9.5 | 7.8 | 5.0 | 4.4 now; 256 rows of 32 000 6.7 and 6.4, fp32 9.3 and 7.9).
template <typename T>
struct Scan {
    static constexpr int VEC = Vec<T>::N;
    const uint4* v4;
    int j_begin, j_end;
    uint4 w[kMonVecs];      // the vectors requested last

    __device__ __forceinline__ void request(int b0) {
#pragma unroll
        for (int u = 0; u < kMonVecs; ++u) {
            const int j = b0 + threadIdx.x + u * kMonThreads;
            w[u] = make_uint4(0, 0, 0, 0);
            if (j < j_end) w[u] = ldg_nc_v4(v4 + j);
        }
    }
    // Requests the first vectors; nothing is waited for.
    __device__ __forceinline__ Scan(const T* row, int begin, int end) : v4(reinterpret_cast<const uint4*>(row)), j_begin(begin), j_end(end) { request(begin); }

    __device__ __forceinline__ Best run(const asynclm_cml_tokens& tok) {
        const int sv[5] = {tok.call / VEC, tok.intr / VEC, tok.trap / VEC, tok.end / VEC, tok.head / VEC};
        auto holds_special = [&](int j) { return j == sv[0] || j == sv[1] || j == sv[2] || j == sv[3] || j == sv[4]; };
        float bv = -INFINITY;
        int bj = -1;
        uint4 bw = make_uint4(0, 0, 0, 0);      // the vector that holds the best value
        for (int b0 = j_begin; b0 < j_end; b0 += kMonVecs * kMonThreads) {
            if (b0 != j_begin) request(b0);
            const int j0 = b0 + threadIdx.x;
            bool special = false;      // does this stretch of vectors hold a CML token? (the same for all threads)
#pragma unroll
            for (int a = 0; a < 5; ++a) special |= (unsigned)(sv[a] - b0) < (unsigned)(kMonVecs * kMonThreads);
#pragma unroll
            for (int u = 0; u < kMonVecs; ++u) {
                const int j = j0 + u * kMonThreads;
                float m = Vec<T>::vmax(w[u]);
                if (special && holds_special(j)) {
                    m = -INFINITY;
#pragma unroll
                    for (int k = 0; k < VEC; ++k)
                        if (!is_special(j * VEC + k, tok)) m = fmaxf(m, Vec<T>::at(w[u], k));
                }
                if (j < j_end && m > bv) { bv = m; bj = j; bw = w[u]; }      // a thread's vectors come in increasing order: the first one wins a tie
            }
        }
        Best best{-INFINITY, INT_MAX};
        if (bj >= 0) {
            const bool mixed = holds_special(bj);
#pragma unroll
            for (int k = VEC - 1; k >= 0; --k)
                if (Vec<T>::at(bw, k) == bv && !(mixed && is_special(bj * VEC + k, tok))) best = Best{bv, bj * VEC + k};
        }
        return best;
    }
};

// CTA-wide best in thread 0 (shuffles inside a warp, shared memory across warps).
__device__ __forceinline__ Best block_best(Best best, float* sv, int* si) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const float v = __shfl_xor_sync(0xffffffffu, best.v, off);
        const int i = __shfl_xor_sync(0xffffffffu, best.i, off);
        if (better(v, i, best)) best = Best{v, i};
    }
    if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = best.v; si[threadIdx.x >> 5] = best.i; }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < kMonThreads / 32; ++w)
            if (better(sv[w], si[w], best)) best = Best{sv[w], si[w]};
    return best;
}

// Grid: (slices, batch).  Every CTA scans one slice of a sequence's row and folds its best ordinary token
// into the row's key with one atomic max; the CTA that arrives last (per-row counter) lets the CML tokens
// that the state allows compete, advances the state machine and puts the two workspace words back to zero.
// The CTAs of a row in the TRAP state read no logits beyond their first request but arrive all the same: state_out may be state_in, so
// nothing is written before every slice of the row has read the state (a CTA arrives behind a block-wide
// barrier, and the two state pointers are not __restrict__).
// The result does not depend on arrival order.  (Scanning all tokens alike and looking at a row a second
// time when a forbidden token had won kept one CTA busy with a whole row after all others had left:
// 256 rows of 128 256 bf16 with a few such rows took 40 us a call on cold inputs, 25 now.)
template <typename T>
__global__ void __launch_bounds__(kMonThreads)
token_monitor_kernel(const T* __restrict__ logits, int vocab, int64_t row_stride, asynclm_cml_tokens tok,
                     const int32_t* state_in, int32_t* __restrict__ token_out,
                     int32_t* state_out, int32_t* __restrict__ flags_out,
                     unsigned long long* __restrict__ ws) {
    constexpr int VEC = Vec<T>::N;
    __shared__ float sv[kMonThreads / 32];
    __shared__ int si[kMonThreads / 32];
    const int seq = blockIdx.y;
    const T* row = logits + (int64_t)seq * row_stride;
    pdl_trigger();      // a kernel behind this one that waits for it may start its prologue
    pdl_wait();         // logits, states and the workspace belong to the kernels in front until those have completed
    const int nvec = vocab / VEC;
    const int per = (nvec + gridDim.x - 1) / gridDim.x;
    const int state = state_in[seq];
    Scan<T> scan(row, blockIdx.x * per, min(nvec, (int)(blockIdx.x + 1) * per));      // on its way beside the state
    // the CML tokens this state allows (INT_MAX: none) and their logits, for the thread that may finish the row
    const int spec0 = state == kText ? tok.call : state == kCall || state == kBody ? tok.end : INT_MAX;
    const int spec1 = state == kText ? tok.trap : state == kCall ? tok.head : INT_MAX;
    float spec_v0 = 0.f, spec_v1 = 0.f;
    Best best{-INFINITY, INT_MAX};
    if (state != kTrap) {
        if (threadIdx.x == 0) {
            if (spec0 != INT_MAX) spec_v0 = to_f32<T>(row[spec0]);
            if (spec1 != INT_MAX) spec_v1 = to_f32<T>(row[spec1]);
        }
        best = scan.run(tok);
        if (blockIdx.x == gridDim.x - 1)      // the row's ragged end, element by element
            for (int i = nvec * VEC + threadIdx.x; i < vocab; i += kMonThreads) {
                const float v = to_f32<T>(row[i]);
                if (!is_special(i, tok) && better(v, i, best)) best = Best{v, i};
            }
        best = block_best(best, sv, si);
    } else {
        __syncthreads();      // every thread has read the state
    }
    if (threadIdx.x != 0) return;
    if (gridDim.x > 1) {
        unsigned long long* key = ws + 2 * (size_t)seq;
        unsigned* arrived = reinterpret_cast<unsigned*>(key + 1);
        if (gridDim.x == 2) {
            // Two slices trade their keys in one atomic, without a counter and the fence in front of it (a round trip each):
            // whoever finds the other's key is the last one.  Its branch on the state is behind it by then, as
            // the other's is behind the trade.
            const unsigned long long mine = best.i != INT_MAX ? pack_key(best.v, best.i) : kNoCandidate, other = atomicExch(key, mine);
            if (other == 0ull) return;
            *key = 0ull;
            best = unpack_key(mine > other ? mine : other);
        } else {
            if (best.i != INT_MAX) atomicMax(key, pack_key(best.v, best.i));
            __threadfence();
            if (atomicAdd(arrived, 1u) != gridDim.x - 1) return;      // not the last CTA of its row
            __threadfence();
            best = unpack_key(atomicExch(key, 0ull));
            *arrived = 0;
        }
    }
    if (state == kTrap) {
        // [TRAP] is followed by [END] whatever the logits say
        token_out[seq] = tok.end;
        state_out[seq] = kText;
        flags_out[seq] = ASYNCLM_MONITOR_TRAP;
        return;
    }
    if (spec0 != INT_MAX && better(spec_v0, spec0, best)) best = Best{spec_v0, spec0};
    if (spec1 != INT_MAX && better(spec_v1, spec1, best)) best = Best{spec_v1, spec1};
    Best pick = best;
    if (pick.i == INT_MAX || pick.v == -INFINITY) {
        // no allowed token has a logit above -inf (all NaN or -inf): the lowest allowed id is taken
        int low = 0;
        while (is_special(low, tok)) ++low;      // lowest ordinary id
        if (state == kText) low = min(low, min(tok.call, tok.trap));
        if (state == kCall) low = min(low, min(tok.head, tok.end));
        if (state == kBody) low = min(low, tok.end);
        pick.i = low;
    }
    int next = state, flags = 0;
    if (state == kText) next = pick.i == tok.call ? kCall : pick.i == tok.trap ? kTrap : kText;
    else if (pick.i == tok.end) { next = kText; flags = ASYNCLM_MONITOR_CALL; }
    else if (state == kCall && pick.i == tok.head) next = kBody;
    if (next == kCall || next == kBody) flags |= ASYNCLM_MONITOR_CRITICAL;
    token_out[seq] = pick.i;
    state_out[seq] = next;
    flags_out[seq] = flags;
}

}  // namespace

}  // namespace asynclm

extern "C" size_t asynclm_token_monitor_workspace_bytes(int32_t batch) { return batch > 0 ? (size_t)batch * 16 : 0; }

extern "C" int asynclm_token_monitor_step(const void* logits, int32_t dtype, int32_t batch, int32_t vocab,
                                          int64_t row_stride, const asynclm_cml_tokens* tokens,
                                          const int32_t* state_in, int32_t* token_out, int32_t* state_out,
                                          int32_t* flags_out, void* workspace, void* stream) {
    using namespace asynclm;
    if (batch < 0 || vocab <= 5 || !tokens || row_stride < vocab || (dtype != ASYNCLM_DTYPE_BF16 && dtype != ASYNCLM_DTYPE_F32))
        return ASYNCLM_ERR_INVALID_ARG;
    if (batch == 0) return ASYNCLM_OK;
    const int ids[5] = {tokens->call, tokens->intr, tokens->trap, tokens->end, tokens->head};
    for (int a = 0; a < 5; ++a) {
        if (ids[a] < 0 || ids[a] >= vocab) return ASYNCLM_ERR_INVALID_ARG;
        for (int b = 0; b < a; ++b) if (ids[a] == ids[b]) return ASYNCLM_ERR_INVALID_ARG;
    }
    const size_t esz = dtype == ASYNCLM_DTYPE_BF16 ? 2 : 4;
    if (!logits || !state_in || !token_out || !state_out || !flags_out || !workspace || ((uintptr_t)logits & 15) != 0 ||
        ((uintptr_t)workspace & 15) != 0 || ((size_t)row_stride * esz) % 16 != 0 || batch > 65535)
        return ASYNCLM_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    // slices per row: about two CTAs per SM in all, at least one pass of kMonVecs vectors per thread each.
    // Fewer, longer CTAs measure faster than many short ones (256 rows of 128 256 bf16: 20.5 us with one
    // or two slices per row, 22.6 with three or four, 24.7 with five to seven): every CTA ends on a
    // block-wide reduction, an atomic and a fence.
    const int nvec = vocab / (16 / (int)esz);
    const int max_slices = std::max(1, nvec / (kMonThreads * kMonVecs));
    const int slices = std::max(1, std::min(max_slices, (148 * 2 + batch - 1) / batch));
    const dim3 grid((unsigned)slices, (unsigned)batch);
    // Launched with programmatic serialization: the launch overlaps the tail of the kernel in front
    // (256 rows of 128 256 bf16, call after call: 16.0 -> 14.6 us, 13.3 with the shorter chain of round trips in each CTA).
    unsigned long long* ws = (unsigned long long*)workspace;
    if (dtype == ASYNCLM_DTYPE_BF16)
        return cuda_status(launch_pdl(token_monitor_kernel<__nv_bfloat16>, grid, dim3(kMonThreads), 0, s, (const __nv_bfloat16*)logits,
                                      vocab, row_stride, *tokens, state_in, token_out, state_out, flags_out, ws));
    return cuda_status(launch_pdl(token_monitor_kernel<float>, grid, dim3(kMonThreads), 0, s, (const float*)logits, vocab, row_stride,
                                  *tokens, state_in, token_out, state_out, flags_out, ws));
}
