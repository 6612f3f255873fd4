// Tensor-core attention for interrupt spans (tcgen05 MMA, accumulators and P in tensor memory).
//
// An interrupt span is a block of new tokens appended to one sequence (paper Section 3.2); in the
// next decoding step (Section 5.3) every token of the span attends to the whole cached context and
// causally to the span itself.  With G query heads per kv head, a span of q tokens gives G*q query
// rows against the same K/V, which is a dense contraction: rows are packed 128 to a tile
// (row r = token r / G, head r % G) and S = Q K^T and O += P V run on the tensor cores.
//
// A work item covers up to 256 query rows (two row tiles) of one (sequence, kv head) and a range of
// keys, 64 to a KV tile.  One persistent CTA per SM, twelve warps:
//   warps 0-3, 4-7  two softmax groups, one thread per query row of a tile.  Each group owns two S
//                   accumulators (64 fp32 columns of tensor memory each) and one O accumulator.
//                     * items with more than 128 rows ("dual"): group b owns row tile b and both
//                       groups consume every KV tile, so K and V are fetched once for 256 rows;
//                     * items with at most 128 rows: the groups take alternate KV tiles of the one
//                       row tile and their (max, sum, O) states are merged in the epilogue like two
//                       KV splits.
//                   The softmax runs in place: a thread reads its row of S and writes P as packed bf16
//                   pairs over columns it has already read; P V then takes its A operand from tensor
//                   memory.  The reference maximum only moves when a score exceeds it by 2^8; then O and
//                   the running sum are rescaled.  The arithmetic around the exponentials is packed two
//                   values to an instruction and reductions run in independent chains.
//                   At the end of an item the rows go out through the group's (now idle) Q tile in
//                   shared memory, so that every global store writes whole 128-byte lines.
//   warps 8, 10     producers of K tiles and of V tiles: one TMA copy a page, completing on the slot's mbarrier (an
//                   unfinished last V page goes row by row through cp.async, with zeros behind the end).  K and V
//                   have a ring of 80 KiB each (see span_ring.h).
//   warps 9, 11     issue the MMAs, one warp per softmax group, by turns.  Warp 9 owns the tensor-memory allocation.
// Why tiles of 64 keys: with two S buffers per group, the Q K^T of the tile after next is issued behind the
// P V of the current one, and the softmax of the next tile, whose S is complete, runs meanwhile; with
// 128-key tiles tensor memory holds one S per group (at head_dim 128) and each group's softmax and MMAs
// took turns.  Per 64 keys of both row tiles (cycles, head_dim 128): the exponential unit needs 1024, the tensor pipe
// 1280 (64-column Q K^T is bound by its operands in shared memory), a lone group's softmax about 1150.
// Why the MMA warps take turns: the pipe serves two warps that issue at once in turn about, so both were done
// at the same time, and then both waited for tiles and scores while the pipe ran dry; the groups' exponentials
// fell together as well.  Turns keep the groups half a period apart.  What a turn has to work out in
// front of its first MMA counts, too: positions in the rings are carried along instead of divided out.
// A tile pair takes 1500-1640 cycles on a CTA alone (2050 with both warps issuing at once and cp.async copies), a
// tile of one row tile 890 (1250; with a copy for each half of a page 1150: see tma_page); at head_dim 64 1520
// (1700) and 900-940 (1070).  When all CTAs stream, the power limit leaves a clock of 1.5-1.7 GHz: attention of 8192 tokens
// of one sequence (32 / 8 heads, head_dim 128) 530-570 -> 490-520 us, 24 sequences with spans of 33-96 tokens over 1-3 K keys
// 82 -> 71-74 us a layer.
// All hand-offs are mbarriers with bounded waits; a wait that runs out sets the plan's status word
// and a CTA-wide abort flag, every role falls through to the common exit, and the tensor memory is
// released there.
#pragma once
#include <cuda.h>

#include <climits>

#include "common.cuh"
#include "kernels.h"
#include "span_ring.h"

namespace asynclm {

namespace tc {

constexpr int kThreads = 384;
constexpr int kProducerWarpK = 8, kMmaWarp = 9, kProducerWarpV = 10;      // 11: the second MMA warp
constexpr int kRows = 128;                       // query rows per row tile
constexpr int kTile = 64;                        // keys per KV tile: a K or V ring slot, an S buffer
constexpr float kRescaleThreshold = 8.f;
constexpr long long kWaitCycles = 2000000000ll;
constexpr long long kGroupSkewCycles = 600;

// Per head_dim: shared memory map (offsets from a 1024-byte aligned base) and barriers.
template <int D>
struct Geometry {
    static constexpr int HALVES = D / 64;                                  // 128-byte pieces of a row
    static constexpr uint32_t QHALF_BYTES = kRows * 128;                   // one 64-value half of a Q tile
    static constexpr uint32_t QTILE_BYTES = HALVES * QHALF_BYTES;
    // A K or V tile is its pages one after the other, a page its two groups of 8 rows, a group its halves of 64 values
    // (8 rows of 128 bytes, swizzled): so one TMA copy lands a whole page, and groups still lie at one stride.
    static constexpr uint32_t ATOM_BYTES = 8 * 128;                        // one half of a group
    static constexpr uint32_t GROUP_BYTES = HALVES * ATOM_BYTES;
    static constexpr uint32_t PAGE_BYTES = 2 * GROUP_BYTES;
    static constexpr uint32_t SLOT_BYTES = kTile / kPage * PAGE_BYTES;
    static constexpr int RING = ring_slots(D);                             // slots of the K ring and of the V ring
    static constexpr uint32_t OFF_Q = 0;                                   // Q[0], Q[1]
    static constexpr uint32_t OFF_RING = OFF_Q + 2 * QTILE_BYTES;
    // The barriers lie behind everything the warp body uses when the CTA goes on to it: arrivals that nobody
    // waits for (an item's last on kOFree and on the ring's empty barriers) may still be queued in the shared
    // memory pipe then, and would change whatever has been copied there since.
    static constexpr uint32_t OFF_BAR = 224 * 1024;
    static_assert(OFF_RING + 2 * RING * SLOT_BYTES <= OFF_BAR, "barriers behind the tiles");
    // S, P and last-P-V hand-offs exist per group b and buffer s: index 2 * b + s
    // (kToken0 + b: it is the turn of group b's MMA warp)
    enum Bar { kQFull = 0, kStats, kOFree, kToken0, kPFull0 = kToken0 + 2, kPvDone0 = kPFull0 + 4, kSFull0 = kPvDone0 + 4,
               kRingFull0 = kSFull0 + 4, kRingEmpty0 = kRingFull0 + 2 * RING, kMmaDrain = kRingEmpty0 + 2 * RING, kNumBars };
    static constexpr uint32_t OFF_TMEM_PTR = OFF_BAR + 8 * kNumBars;
    static constexpr uint32_t OFF_ABORT = OFF_TMEM_PTR + 8;
    static constexpr uint32_t SMEM_BYTES = OFF_ABORT + 8 + 1024;
    static_assert(SMEM_BYTES <= 232448, "shared memory budget");
};

// tensor memory columns
constexpr uint32_t kColS = 0;      // S[b][s]: 64 columns each at 128 b + 64 s; P[b][s] overlays the first 32 of S[b][s]
constexpr uint32_t kColO = 256;    // O[b]: head_dim columns each
constexpr uint32_t kTmemCols = 512;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int32_t* status, int code) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        __nanosleep(32);      // leave the issue slots to the warps that have work
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort_flag = 1;
            atomicCAS(status, 0, code);
            return false;
        }
    }
    return true;
}
// The same wait without the back-off, for the one thread that issues the MMAs: what it waits for is on
// the critical path of both softmax groups.
__device__ __forceinline__ bool mbar_wait_spin(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int32_t* status, int code) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort_flag = 1;
            atomicCAS(status, 0, code);
            return false;
        }
    }
    return true;
}
// The same wait with a warp-uniform verdict, for code that goes on to warp-collective instructions.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int32_t* status, int code) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status, code));
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros instead.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
// Arrive on the mbarrier once all cp.async copies issued so far by this thread have landed.
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// A page's 16 K or V rows of one kv head, `block` = (2 * page + K|V) * Hkv + head, land as [2 groups of 8 rows][halves]
// [8 rows][128 bytes], 16-byte pieces XOR-swizzled by row (see make_pool_map).  One SM's TMA unit takes about as long
// for a copy of 2 KB (35 ns) as for one of 4 KB (44 ns): with a copy for each half of a page, one SM
// streamed 57 KB/us, with one for both 92.  No multicast.
__device__ __forceinline__ void tma_page(uint32_t dst, const CUtensorMap* map, int block, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(map), "r"(0), "r"(0), "r"(0), "r"(0), "r"(block), "r"(bar) : "memory");
}

// Shared-memory matrix descriptor, 128-byte swizzle, descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
    return (uint64_t)((addr & 0x3ffffu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) |
           ((uint64_t)(sbo_bytes >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = n; b_mn = 1 when B is stored with N
// contiguous (the V tile), 0 when K is contiguous.
__host__ __device__ constexpr uint32_t instr_desc(uint32_t n, uint32_t b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn << 16) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
// `el`: 1 in the lane that issues, 0 in the others (the warp stays converged, so that operands are uniform).
__device__ __forceinline__ void mma_f16(uint32_t el, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"(el) : "memory");
}
// True in exactly one lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\tselp.u32 %0, 1, 0, e;\n\t}" : "=r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void mma_commit(uint32_t el, uint32_t bar) {
    asm volatile("{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %1, 0;\n\t"
                 "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(el) : "memory");
}

#define TC_R32(r) \
    "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), \
    "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), \
    "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), \
    "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
#define TC_W32(r) \
    "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), \
    "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), \
    "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), \
    "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])

// This warp's 32 rows x 32 consecutive fp32 columns of tensor memory -> one row per thread.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : TC_R32(r) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31};"
        ::TC_W32(r), "r"(taddr) : "memory");
}
// Waits for this thread's tensor-memory loads; the loaded registers pass through the statement so that
// no use of them can be scheduled in front of it.
__device__ __forceinline__ void tmem_wait_ld_dep(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 16 consecutive 32-bit columns of this warp's 32 rows.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};"
        ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t& a, uint32_t& b) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(a), "=r"(b) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st2(uint32_t taddr, uint32_t a, uint32_t b) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%2], {%0,%1};" ::"r"(a), "r"(b), "r"(taddr) : "memory");
}
// D (+)= A B with A taken from tensor memory: row i of A is lane i, its 16 bf16 values of one K step
// are 8 consecutive 32-bit columns (two values per column, the lower index in the low half).
__device__ __forceinline__ void mma_f16_ta(uint32_t el, uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(acc), "r"(el) : "memory");
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// One work item as the kernel sees it (kv_end == 0: no item).
struct TItem {
    int kv0, kv_end, q_row0, ntok, kv_limit0, kv_head, partial_row0, page0;
};

// `rec`: a Work record (the planner's array, or the copy of a CTA's first item in its header).
__device__ __forceinline__ TItem load_titem(const Work* rec, bool valid) {
    TItem r{0, 0, 0, 0, 0, 0, -1, 0};
    if (valid) {
        const int4* src = reinterpret_cast<const int4*>(rec);
        const int4 a = __ldg(src), b = __ldg(src + 1);
        r.kv0 = a.x; r.kv_end = a.y; r.q_row0 = a.z; r.ntok = a.w;
        r.kv_limit0 = b.x; r.kv_head = b.y; r.partial_row0 = b.z; r.page0 = b.w;
    }
    return r;
}

// The whole kernel body, called by all twelve warps with `smem` 1024-byte aligned.
// ALONE: in the kernel of steps that have span tiles only.  A launch starts on cold instruction caches, and there every line
// of code that is fetched for the first time stands in the way: the P V of an unfinished last tile is a loop, and the output rows
// go out in two passes of four at head_dim 128 (at 64, where a warp has one or two slices, two passes are slower).  us of
// attention, unrolled | so, before the tiles came by TMA in brackets: 4 sequences of 100-300 keys with spans of 20-60 tokens
// 14.04 | 13.68 (14.04), one span over 2000 keys 15.6 | 15.1 (15.2), head_dim 64 9.57 | 9.47 (9.18), 24 sequences with spans of 33-96
// tokens 70.3 | 69.1, 8192 tokens 545 | 528.  Beside the warp body's code it is a loss: 8 sequences of 32-131 K keys with two
// 256-token spans 917 | 925.
template <int D, int G, bool ALONE>
__device__ __forceinline__ void tc_body(const DevPlan& p, const CUtensorMap* span_map, const __nv_bfloat16* __restrict__ q,
                                        const __nv_bfloat16* pool,
                                        __nv_bfloat16* __restrict__ out, float* __restrict__ lse,
                                        uint8_t* smem) {
    using Geo = Geometry<D>;
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + Geo::OFF_BAR;
    auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
    volatile uint32_t* tmem_ptr = (volatile uint32_t*)(smem + Geo::OFF_TMEM_PTR);
    volatile int* abort_flag = (volatile int*)(smem + Geo::OFF_ABORT);

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int Hq = p.num_q_heads, Hkv = p.num_kv_heads;
    // The plan is there when this kernel starts (behind an upload by kernel the first launch starts when that has completed: PlanUse),
    // so it may be read before pdl_wait(); everything else (pool, q, outputs) is touched only after it.
    const int32_t* head = p.cta_heads + (size_t)blockIdx.x * kHeadWords;
    const int i0 = head[0], i1 = head[1];
    const Work* head_work = reinterpret_cast<const Work*>(head + kHeadWorkTensor);      // = p.works[i0]

    if (threadIdx.x == 0) {
        mbar_init(bar(Geo::kQFull), 256);
        mbar_init(bar(Geo::kStats), 256);
        mbar_init(bar(Geo::kOFree), 256);
        mbar_init(bar(Geo::kToken0), 1);
        mbar_init(bar(Geo::kToken0 + 1), 1);
        for (int b = 0; b < 4; ++b) {
            mbar_init(bar(Geo::kPFull0 + b), 4);      // one arrival per warp of the group
            mbar_init(bar(Geo::kPvDone0 + b), 1);
            mbar_init(bar(Geo::kSFull0 + b), 1);
        }
        for (int s = 0; s < 2 * Geo::RING; ++s) {
            mbar_init(bar(Geo::kRingFull0 + s), s < Geo::RING ? 1 : 33);      // V tiles: see the producers
            mbar_init(bar(Geo::kRingEmpty0 + s), 2);
        }
        mbar_init(bar(Geo::kMmaDrain), 2);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (threadIdx.x == kProducerWarpK * 32) asm volatile("prefetch.tensormap [%0];" ::"l"(span_map));
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(sbase + Geo::OFF_TMEM_PTR), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_ptr;

    if (warp >= 8) {
      if (warp == kProducerWarpK || warp == kProducerWarpV) {
        // ------------------------------------------------------------------ producer warps
        const int which = warp == kProducerWarpV ? 1 : 0;       // 0: K tiles, 1: V tiles
        const uint32_t ring = sbase + Geo::OFF_RING;
        auto load_pages = [&](const TItem& it, int first_page) {
            const int npg = (it.kv_end - it.kv0 + kPage - 1) / kPage;
            const int idx = first_page + lane;
            return idx < npg ? __ldg(p.page_indices + it.page0 + idx) : 0;
        };
        auto land_copies = [&](int k0, int k1) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            const long long t0 = clock64();
            for (int k = k0; k < k1; ++k)
                while (!mbar_try_wait(bar(Geo::kRingFull0 + ring_slot(which, k, Geo::RING)), (uint32_t)ring_use(k, Geo::RING) & 1u) &&
                       clock64() - t0 < kWaitCycles) {}
        };
        constexpr int kPagesPerTile = kTile / kPage;          // 4
        constexpr int kGroupTiles = 32 / kPagesPerTile;       // 8
        constexpr int kChunks = D / 8, kRowsPerOp = 32 / kChunks;      // cp.async: 16-byte chunks of a row; rows a warp instruction moves
        bool ok = true;
        int n = 0;                                             // tiles issued so far (all items)
        int ev = 0;      // time-stamp build: event log position (lane 0 of a producer)
        TItem cur = load_titem(head_work, i0 < i1), nxt = load_titem(p.works + i0 + 1, i0 + 1 < i1);
        int pages_cur = head[kHeadPagesTensor + lane];      // the first item's first 32 page ids (0 beyond its end)
        pdl_wait();
        for (int ii = i0; cur.kv_end > 0 && ok; ++ii) {
            const TItem after = load_titem(p.works + ii + 2, ii + 2 < i1);
            const int ntiles = (cur.kv_end - cur.kv0 + kTile - 1) / kTile;
            for (int t0 = 0; t0 < ntiles && ok; t0 += kGroupTiles) {
                int pages_nxt = 0;
                const int t1 = min(t0 + kGroupTiles, ntiles);
                for (int t = t0; t < t1 && ok; ++t, ++n) {
                    const int rows = min(kTile, cur.kv_end - (cur.kv0 + t * kTile));
                    const int npages = (rows + kPage - 1) / kPage;
                    const int s = ring_slot(which, n, Geo::RING);
                    if (lane == 0 && which == 0) trace_event(9, ev, 40);
                    ok = mbar_wait_warp(bar(Geo::kRingEmpty0 + s), ((uint32_t)ring_use(n, Geo::RING) & 1u) ^ 1u, abort_flag, p.status, 11 + which);
                    if (!ok) break;
                    if (lane == 0 && which == 0) trace_event(9, ev, 42);
                    const uint32_t full = bar(Geo::kRingFull0 + s), slot_addr = ring + s * Geo::SLOT_BYTES;
                    // Slots past the item's end hold anything.  K's only reach scores that the softmax masks, but 0 * NaN
                    // would poison P V, so the item's last V page, if it is not full, is copied row by row with zeros
                    // behind the end.  A V barrier takes 33 arrivals: one with the byte count of the TMA copies, and one
                    // of each lane's cp.async copies or all 32 at once where there are none.
                    const bool ragged = which == 1 && last_page_by_rows(cur.kv_end, t == ntiles - 1, kPage);
                    const int npages_tma = npages - (ragged ? 1 : 0);
#ifdef ASYNCLM_DEBUG
                    // checked build: a test may ask for one hand-off to be left out, to see a bounded wait run out
                    const bool stall = which == 0 && blockIdx.x == 0 && p.debug_stall_tile == n + 1;
#else
                    constexpr bool stall = false;
#endif
                    if (lane == 0 && !stall) {
                        mbar_arrive_expect_tx(full, (uint32_t)npages_tma * Geo::PAGE_BYTES);
                        if (which == 1 && !ragged) mbar_arrive_n(full, 32);
                    }
                    __syncwarp();
                    int page = __shfl_sync(0xffffffffu, pages_cur, (t - t0) * kPagesPerTile + min(lane, npages - 1));
                    // checked build only: a bad id is replaced by page 0 (the copy must happen: the barrier counts its bytes)
                    if (lane < npages && !page_ok(page, p.num_pages, p.status, kStatusBadPageSpan)) page = 0;
                    if (lane < npages_tma && !stall)
                        tma_page(slot_addr + (uint32_t)lane * Geo::PAGE_BYTES, span_map, (2 * page + which) * Hkv + cur.kv_head, full);
                    if (ragged) {
                        page = __shfl_sync(0xffffffffu, page, npages - 1);
                        const uint8_t* src_page = reinterpret_cast<const uint8_t*>(pool + pool_row_offset(page, which, cur.kv_head, 0, Hkv, D));
                        // lane -> 16-byte chunk c of a row: a warp instruction moves whole rows, 512 bytes in all
                        const int c = lane % kChunks;
#pragma unroll
                        for (int rr = 0; rr < kPage / kRowsPerOp; ++rr) {
                            const int slot = rr * kRowsPerOp + lane / kChunks;
                            cp_async16(slot_addr + (uint32_t)(npages - 1) * Geo::PAGE_BYTES + (uint32_t)(slot >> 3) * Geo::GROUP_BYTES +
                                           (uint32_t)(c >> 3) * Geo::ATOM_BYTES + (uint32_t)(slot & 7) * 128u + (uint32_t)(((c & 7) ^ (slot & 7)) << 4),
                                       src_page + slot * (D * 2) + c * 16, (npages - 1) * kPage + slot < rows ? 16u : 0u);
                        }
                        cp_async_arrive(full);
                    }
                    if (lane == 0 && which == 0) trace_event(9, ev, 44);
                    // page ids of the next group of tiles (or of the next item), requested only after this
                    // group's first tile is on its way: the next item's descriptor may still be in flight
                    if (t == t0) {
                        if (t0 + kGroupTiles < ntiles) pages_nxt = load_pages(cur, (t0 + kGroupTiles) * kPagesPerTile);
                        else if (nxt.kv_end > 0) pages_nxt = load_pages(nxt, 0);
                    }
                }
                pages_cur = pages_nxt;
            }
            cur = nxt;
            nxt = after;
        }
        // The copies land before shared memory goes away or on to the warp body.  The MMA warps have normally waited for
        // each of them, but another role may have given up meanwhile, whether or not this one has seen it.
        land_copies(max(0, n - Geo::RING), n);
      } else {
        // ------------------------------------------------------------------ MMA issuers
        // One warp per softmax group, running convergently, issues the group's MMAs through an elected lane.  A
        // turn is one KV tile of the group: its P V and the Q K^T of the group's next tile
        // but one into the S buffer that the P V has just read (MMAs of one thread execute in issue order).
        // While the tensor core works on a turn, the group runs the softmax of its other buffer: neither
        // waits for the other as long as both keep up.
        const int b = warp == kMmaWarp ? 0 : 1;
        const uint32_t el = elect_one() ? 1u : 0u;
        bool ok = true;
        int base = 0;             // KV tiles before this item
        int cnt = 0;              // tiles of the group before this item: S buffer and phase of the hand-offs
        int item_no = 0;
        // The warps take turns, group 0 first, whether they have MMAs to issue or not: turn n of warp 1 follows turn n of
        // warp 0, turn n of warp 0 follows turn n - 1 of warp 1.  Not only for speed: a turn's waits for tiles stand in front of its
        // token, and that order is what makes the parities of the ring's full barriers unambiguous (see span_ring.h).
        int turn_no = 0;
        auto take_token = [&](bool& good) {
            good = good && (b + turn_no == 0 || mbar_wait_spin(bar(Geo::kToken0 + b), (uint32_t)(turn_no + b + 1) & 1u, abort_flag, p.status, 28));
            ++turn_no;
        };
        auto pass_token = [&]() { if (lane == 0) mbar_arrive(bar(Geo::kToken0 + (b ^ 1))); };
        constexpr uint32_t idesc_pv = instr_desc(D, 1);
        const uint32_t ocol = tmem + kColO + (uint32_t)(D * b);
        TItem it_next = load_titem(head_work, i0 < i1);
        const long long t_loop = trace_clock();
        long long tr_p = 0, tr_kv = 0, tr_item = 0;      // time-stamp build: cycles waiting for P, for K/V, for an item's Q and O
        int ev = 0;                                      // time-stamp build: event log position
        for (int ii = i0; ii < i1 && ok; ++ii, ++item_no) {
            const TItem it = it_next;
            it_next = load_titem(p.works + ii + 1, ii + 1 < i1);      // in flight while this item runs
            const int ntiles = (it.kv_end - it.kv0 + kTile - 1) / kTile;
            const bool dual = it.ntok * G > kRows;      // both groups on every tile, group b on row tile b; otherwise alternate tiles
            const int lead = dual ? 2 : 4, mine = dual ? ntiles : (ntiles + 1 - b) / 2;
            const long long t_item = trace_clock();
            ok = mbar_wait_spin(bar(Geo::kQFull), (uint32_t)item_no & 1u, abort_flag, p.status, 22);
            // S and O of the previous item are in use until its epilogue is over
            if (ok && item_no > 0) ok = mbar_wait_spin(bar(Geo::kOFree), (uint32_t)(item_no - 1) & 1u, abort_flag, p.status, 27);
            tr_item += trace_clock() - t_item;
            if (ok) tc_fence_after();
            const uint64_t qd = smem_desc(sbase + Geo::OFF_Q + (dual ? (uint32_t)b * Geo::QTILE_BYTES : 0u), 16, 1024);
            const int last_pages = (it.kv_end - (it.kv0 + (ntiles - 1) * kTile) + kPage - 1) / kPage;      // of the item's last tile
            const uint32_t idesc_last = instr_desc(16u * (uint32_t)last_pages, 0);
            // where the group's next K and V tile lie
            RingPlace kp = ring_place(base + (dual ? 0 : b), Geo::RING), vp = kp;
            auto next_place = [&](RingPlace& x) { x = ring_next(x, dual ? 1 : 2, Geo::RING); };
            auto wait_tile = [&](int which, const RingPlace& x, int code) {
                const long long tw = trace_clock();
                ok = ok && mbar_wait_spin(bar(Geo::kRingFull0 + which * Geo::RING + x.slot), x.parity, abort_flag, p.status, code);
                tr_kv += trace_clock() - tw;
            };
            auto tile_addr = [&](int which, const RingPlace& x) { return sbase + Geo::OFF_RING + (uint32_t)(which * Geo::RING + x.slot) * Geo::SLOT_BYTES; };
            // u = -2, -1: the Q K^T of the group's first two tiles; u >= 0: the turn of its u-th tile, the P V of
            // tile j and the Q K^T of tile j + lead back to back once everything they read is there.  K/V tiles
            // are waited for first (they are normally there already), P last, so that nothing stands between
            // its arrival and the first MMA.  One commit per turn: it tells the group that its next S is complete
            // and, because MMAs complete in issue order, that every MMA in front of it is done as well (the
            // group releases ring slots on that knowledge; a commit costs the tensor pipe ~90 cycles).  Where no
            // next tile is left the P V is committed by itself: the last turn on either buffer ends on kPvDone.
            for (int u = -2; u < mine && ok; ++u) {
                const int c = cnt + u;
                const bool pv = u >= 0, qk = u + 2 < mine;
                if (!pv && !qk) {
                    take_token(ok);
                    pass_token();
                    continue;
                }
                const int j = dual ? u : 2 * u + b, jn = j + lead;
                if (lane == 0) trace_event(b ? 10 : 0, ev, 20 + b);
                if (pv) wait_tile(1, vp, 24);
                if (qk) wait_tile(0, kp, 21);
                // The tiles were written by TMA copies, but for the rows of an unfinished last V page: those came by cp.async,
                // through the generic proxy, and the MMAs read through the asynchronous one.  The full barrier orders
                // the two, the fence makes the bytes visible across.
                if (pv && last_page_by_rows(it.kv_end, j == ntiles - 1, kPage)) fence_async_smem();
                const uint32_t buf = tmem + kColS + 128u * (uint32_t)b + 64u * (uint32_t)(c & 1);      // S and P
                const uint64_t vd = smem_desc(tile_addr(1, vp), Geo::ATOM_BYTES, Geo::GROUP_BYTES);
                const uint64_t kd = smem_desc(tile_addr(0, kp), 16, Geo::GROUP_BYTES);
                const uint32_t idesc_qk = jn == ntiles - 1 ? idesc_last : instr_desc(kTile, 0);
                const uint32_t done = bar((qk ? Geo::kSFull0 : Geo::kPvDone0) + 2 * b + (c & 1));
                if (pv) {
                    const long long tw = trace_clock();
                    ok = ok && mbar_wait_spin(bar(Geo::kPFull0 + 2 * b + (c & 1)), (uint32_t)(c >> 1) & 1u, abort_flag, p.status, 26);
                    tr_p += trace_clock() - tw;
                }
                take_token(ok);
                if (lane == 0) trace_event(b ? 10 : 0, ev, 22 + b);
                if (!ok) break;
                tc_fence_after();
                if (pv) {
                    // O[b] (+)= P[b] V_j with P[b] in tensor memory
                    if (j < ntiles - 1 || last_pages == kTile / kPage) {
#pragma unroll
                        for (int ks = 0; ks < kTile / kPage; ++ks)
                            mma_f16_ta(el, ocol, buf + 8u * (uint32_t)ks, vd + (uint64_t)ks * (Geo::PAGE_BYTES >> 4), idesc_pv, (u > 0 || ks > 0) ? 1u : 0u);
                    } else if constexpr (ALONE) {
#pragma unroll 1
                        for (int ks = 0; ks < last_pages; ++ks)
                            mma_f16_ta(el, ocol, buf + 8u * (uint32_t)ks, vd + (uint64_t)ks * (Geo::PAGE_BYTES >> 4), idesc_pv, (u > 0 || ks > 0) ? 1u : 0u);
                    } else {
                        for (int ks = 0; ks < last_pages; ++ks)
                            mma_f16_ta(el, ocol, buf + 8u * (uint32_t)ks, vd + (uint64_t)ks * (Geo::PAGE_BYTES >> 4), idesc_pv, (u > 0 || ks > 0) ? 1u : 0u);
                    }
                }
                if (qk) {
                    // S[b] <- Q[b] K^T
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks) {
                        if (ks == D / 16 - 2) pass_token();      // the other warp's first MMA queues behind the last two
                        // the address field counts 16-byte units and cannot carry out of its 14 bits here
                        const uint64_t qoff = (uint64_t)(((uint32_t)(ks >> 2) * Geo::QHALF_BYTES + (uint32_t)(ks & 3) * 32u) >> 4);
                        const uint64_t koff = (uint64_t)(((uint32_t)(ks >> 2) * Geo::ATOM_BYTES + (uint32_t)(ks & 3) * 32u) >> 4);
                        mma_f16(el, buf, qd + qoff, kd + koff, idesc_qk, ks > 0);
                    }
                }
                mma_commit(el, done);
                if (!qk) pass_token();
                if (pv) next_place(vp);
                if (qk) next_place(kp);
                if (lane == 0) trace_event(b ? 10 : 0, ev, 26 + b);
            }
            if (!dual && b == 1 && (ntiles & 1) != 0) {      // group 0 has a turn more
                take_token(ok);
                pass_token();
            }
            cnt += mine;
            base += ntiles;
        }
        if (lane == 0 && b == 0) {
            trace_set(8, tr_p);
            trace_set(9, tr_kv);
            trace_set(10, trace_clock() - t_loop);
            trace_set(14, tr_item);
        }
        // make sure nothing is still running on the tensor core before tensor memory is released
        mma_commit(el, bar(Geo::kMmaDrain));
        const long long t0 = clock64();
        while (!mbar_try_wait(bar(Geo::kMmaDrain), 0) && clock64() - t0 < kWaitCycles) {}
        __syncwarp();
      }
    } else {
        // ------------------------------------------------------------------ softmax / epilogue groups
        const int b = warp >> 2;                   // softmax group
        const int m = threadIdx.x & 127;           // row of the group's tile = tensor-memory lane
        const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t s_addr = lane_addr + kColS + 128u * (uint32_t)b;      // + 64 * buffer
        const uint32_t o_addr = lane_addr + kColO + (uint32_t)(D * b);
        const float qscale = p.sm_scale * kLog2e;
        const float2 qscale2 = make_float2(qscale, qscale);
        int cnt = 0;         // tiles this group has processed before this item
        int kv_base = 0;     // KV tiles of the CTA before this item (both groups)
        uint32_t pv_phase = 0;      // bit s: parity of the next phase of this group's kPvDone of buffer s
        int item_no = 0;
        bool ok = true;
        long long tr_wait = 0, tr_work = 0, tr_tiles = 0;      // time-stamp build: cycles waiting for S, cycles from S to P, tiles
        int ev = 0;                                            // time-stamp build: event log position (lane 0 of each warp)
        // This thread's share of an item's Q.  Dual items: the whole row 128 b + m (kQV chunks of 16
        // bytes) into Q[b]; otherwise value half b of row m (kQV / 2 chunks) into Q[0].  The next item's Q is
        // fetched at the end of the current item's KV loop, ahead of the epilogue.
        constexpr int kQV = D / 8;
        auto load_q = [&](const TItem& x, uint4 (&w)[kQV]) {
            const bool dual = x.ntok * G > kRows;
            const int r = dual ? 128 * b + m : m;
            const bool valid = x.kv_end > 0 && r / G < x.ntok;
            const uint4* src = reinterpret_cast<const uint4*>(
                q + ((size_t)(x.q_row0 + r / G) * Hq + (size_t)x.kv_head * G + r % G) * D) + (dual ? 0 : kQV / 2 * b);
#pragma unroll
            for (int c = 0; c < kQV / 2; ++c) w[c] = valid ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int c = kQV / 2; c < kQV; ++c) w[c] = (valid && dual) ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
        };
        // A ring slot is free again after two arrivals: one of each group in a dual item, else two of its only reader.
        auto release = [&](int which, int t, bool dual) { mbar_arrive_n(bar(Geo::kRingEmpty0 + ring_slot(which, t, Geo::RING)), dual ? 1u : 2u); };
        TItem it_next = load_titem(head_work, i0 < i1);
        uint4 q_next[kQV];
        pdl_wait();
        load_q(it_next, q_next);
        for (int ii = i0; ii < i1 && ok; ++ii, ++item_no) {
            const TItem it = it_next;
            const int ntiles = (it.kv_end - it.kv0 + kTile - 1) / kTile;
            const bool dual = it.ntok * G > kRows;
            const int lead = dual ? 2 : 4;
            const int mine = dual ? ntiles : (ntiles + 1 - b) / 2;      // KV tiles of this group
            const int r = dual ? 128 * b + m : m;      // query row of the item
            const int t = r / G, g = r % G;
            const bool row_valid = t < it.ntok;
            // ---- stage Q with the 128-byte swizzle the MMA descriptor expects (the previous item's
            // epilogue used the Q tiles as its output staging area: wait until every warp is through)
            if (item_no > 0) {
                ok = mbar_wait_warp(bar(Geo::kOFree), (uint32_t)(item_no - 1) & 1u, abort_flag, p.status, 36);
                if (!ok) break;
            }
#pragma unroll
            for (int c = 0; c < kQV; ++c)
                if (dual || c < kQV / 2) {
                    const int cc = dual ? c : c + kQV / 2 * b;      // chunk of the row
                    *reinterpret_cast<uint4*>(smem + Geo::OFF_Q + (dual ? b * Geo::QTILE_BYTES : 0u) + (cc >> 3) * Geo::QHALF_BYTES + m * 128 +
                                              (((cc & 7) ^ (m & 7)) << 4)) = q_next[c];
                }
            fence_async_smem();
            mbar_arrive(bar(Geo::kQFull));
            if (lane == 0) trace_event(1 + warp, ev, 37);
            it_next = load_titem(p.works + ii + 1, ii + 1 < i1);
            const int lim_row = row_valid ? min(it.kv_limit0 + t, it.kv_end) : 0;   // keys [0, lim_row) visible
            float m_ref = -INFINITY;                     // reference maximum (log2 domain)
            float2 l2 = make_float2(0.f, 0.f), l2b = make_float2(0.f, 0.f);      // running sum of P, four partial sums
            for (int u = 0; u < mine && ok; ++u) {
                const int j = dual ? u : 2 * u + b, ct = cnt + u;
                const int npg = (min(kTile, it.kv_end - (it.kv0 + j * kTile)) + kPage - 1) / kPage;
                const uint32_t sb = s_addr + 64u * (uint32_t)(ct & 1);
                const long long tw = trace_clock();
                if (lane == 0) trace_event(1 + warp, ev, 30);
                ok = __all_sync(0xffffffffu, mbar_wait_spin(bar(Geo::kSFull0 + 2 * b + (ct & 1)), (uint32_t)(ct >> 1) & 1u, abort_flag, p.status, 31));
                const long long ts = trace_clock();
                if (lane == 0) trace_event(1 + warp, ev, 31);
                tr_wait += ts - tw;
                ++tr_tiles;
                if (!ok) break;
                tc_fence_after();
                const int base = it.kv0 + j * kTile;
                const int vis = max(0, min(kTile, lim_row - base));      // visible columns of this row
                uint32_t rr[64];
                tmem_ld32(sb, *reinterpret_cast<uint32_t(*)[32]>(&rr[0]));
                tmem_ld32(sb + 32u, *reinterpret_cast<uint32_t(*)[32]>(&rr[32]));
                // This S complete means every MMA issued for the group before it is complete: the ring slots they
                // read go back to the producers, the K tile of j now, and the V tile of j - lead (its P V was
                // issued in front of this Q K^T).
                if (m == 0) {
                    release(0, kv_base + j, dual);
                    if (u >= 2) release(1, kv_base + j - lead, dual);
                }
                tmem_wait_ld();
                if (!__all_sync(0xffffffffu, vis == kTile)) {
#pragma unroll
                    for (int e = 0; e < 64; ++e)
                        if (e >= vis) rr[e] = 0xff800000u;      // -inf
                }
                // row maximum of the raw scores (the scale is positive): four independent chains of 3-input
                // maxima (a lone warp per scheduler cannot hide one long dependent chain)
                auto sv = [&](int k) { return __uint_as_float(rr[k]); };
                float cm[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) cm[c] = fmax3(sv(16 * c), sv(16 * c + 1), sv(16 * c + 2));
#pragma unroll
                for (int k = 3; k < 15; k += 2) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) cm[c] = fmax3(cm[c], sv(16 * c + k), sv(16 * c + k + 1));
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) cm[c] = fmaxf(cm[c], sv(16 * c + 15));
                const float cmax = fmax3(fmaxf(cm[0], cm[1]), cm[2], cm[3]) * qscale;      // log2 domain
                if (__any_sync(0xffffffffu, cmax > m_ref + kRescaleThreshold)) {
                    // Move the reference maximum (rare after the first tile; a row without one takes any visible
                    // key's): rescale the running sum and O[b].  O[b] is at rest once the P V of the group's
                    // previous tile is done, which its commit tells: the next S of the other buffer, or kPvDone.
                    const float m_new = fmaxf(m_ref, cmax);
                    const float scale = m_new == -INFINITY ? 1.f : fast_exp2(m_ref - m_new);
                    m_ref = m_new;
                    l2.x *= scale;
                    l2.y *= scale;
                    l2b.x *= scale;
                    l2b.y *= scale;
                    if (u > 0) {
                        const int ob = (ct + 1) & 1, pb = (u + 1 < mine ? Geo::kSFull0 : Geo::kPvDone0) + 2 * b + ob;
                        const uint32_t pp = u + 1 < mine ? (uint32_t)((ct + 1) >> 1) & 1u : (pv_phase >> ob) & 1u;
                        ok = __all_sync(0xffffffffu, mbar_wait_spin(bar(pb), pp, abort_flag, p.status, 32));
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll 1
                        for (int cc = 0; cc < D / 16; ++cc) {
                            uint32_t ro[16];
                            tmem_ld16(o_addr + 16u * cc, ro);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 16; ++e) ro[e] = __float_as_uint(__uint_as_float(ro[e]) * scale);
                            tmem_st16(o_addr + 16u * cc, ro);
                        }
                        tmem_wait_st();
                    }
                }
                // Both groups of a dual item get their first S together and would stay in step, both on the
                // exponential unit at once and both off it: the second group starts half a tile later.
                if (dual && b == 1 && u == 0) {
                    const long long t0 = clock64();
                    while (clock64() - t0 < kGroupSkewCycles) {}
                }
                // P = exp2(S * scale - m_ref) as packed bf16 goes to the first 32 columns of the buffer, which this
                // thread has read
                const float m_use = m_ref == -INFINITY ? 0.f : m_ref;
                const float2 nm2 = make_float2(-m_use, -m_use);
                uint32_t pk[32];
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    const float2 x = __ffma2_rn(make_float2(__uint_as_float(rr[2 * e]), __uint_as_float(rr[2 * e + 1])), qscale2, nm2);
                    const float2 pe = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                    if (e & 1) l2b = __fadd2_rn(l2b, pe); else l2 = __fadd2_rn(l2, pe);
                    pk[e] = pack_bf16x2(pe.x, pe.y);
                }
                tmem_st16(sb, *reinterpret_cast<uint32_t(*)[16]>(&pk[0]));
                tmem_st16(sb + 16u, *reinterpret_cast<uint32_t(*)[16]>(&pk[16]));
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();      // 128 arrivals on one barrier word would take turns; the warp's lanes are ordered here instead
                if (lane == 0) mbar_arrive(bar(Geo::kPFull0 + 2 * b + (ct & 1)));
                tr_work += trace_clock() - ts;
                if (lane == 0) trace_event(1 + warp, ev, 32);
            }
            if (!ok) break;
            const float l_sum = (l2.x + l2.y) + (l2b.x + l2b.y);
            load_q(it_next, q_next);        // in flight during the epilogue
            if (lane == 0) trace_event(1 + warp, ev, 33);
            // ---- epilogue.  The groups' (max, sum) go through columns 0-1 of their S buffers, which are
            // idle from the group's last P V until the next item's first Q K^T.
            for (int u = max(0, mine - 2); u < mine && ok; ++u) {
                const int sb = (cnt + u) & 1;
                ok = mbar_wait_warp(bar(Geo::kPvDone0 + 2 * b + sb), (pv_phase >> sb) & 1u, abort_flag, p.status, 34);
                pv_phase ^= 1u << sb;
                // the V tiles of the group's last tiles go back to the producers
                if (ok && m == 0) release(1, kv_base + (dual ? u : 2 * u + b), dual);
            }
            if (!ok) break;
            tc_fence_after();
            if (lane == 0) trace_event(1 + warp, ev, 34);
            tmem_st2(s_addr, __float_as_uint(m_ref), __float_as_uint(l_sum));
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar(Geo::kStats));
            ok = mbar_wait_warp(bar(Geo::kStats), (uint32_t)item_no & 1u, abort_flag, p.status, 35);
            if (!ok) break;
            tc_fence_after();
            if (lane == 0) trace_event(1 + warp, ev, 35);
            const size_t hq = (size_t)it.kv_head * G + g;
            const size_t prow = it.partial_row0 < 0 ? 0 : (size_t)it.partial_row0 + t;
            float w0, w1, lse2;          // weights of O[0] and O[1] in this thread's output row
            int c_begin, c_end;          // 32-column chunks of the row this thread writes
            if (dual) {
                const float inv = l_sum > 0.f ? 1.f / l_sum : 0.f;
                w0 = b == 0 ? inv : 0.f;
                w1 = b == 1 ? inv : 0.f;
                lse2 = l_sum > 0.f ? m_ref + log2f(l_sum) : -INFINITY;
                c_begin = 0; c_end = D / 32;
            } else {
                // the two groups hold two KV splits of the same rows: merge them; a group writes slices of 64 values,
                // group b the b-th (head_dim 64 has only one)
                uint32_t x0, y0, x1, y1;
                tmem_ld2(lane_addr + kColS, x0, y0);
                tmem_ld2(lane_addr + kColS + 128u, x1, y1);
                tmem_wait_ld();
                const float m0 = __uint_as_float(x0), l0 = __uint_as_float(y0);
                const float m1 = __uint_as_float(x1), l1 = __uint_as_float(y1);
                const float M = fmaxf(m0, m1);
                const float a0 = l0 > 0.f ? fast_exp2(m0 - M) : 0.f;
                const float a1 = l1 > 0.f ? fast_exp2(m1 - M) : 0.f;
                const float L = a0 * l0 + a1 * l1;
                const float inv = L > 0.f ? 1.f / L : 0.f;
                w0 = a0 * inv;
                w1 = a1 * inv;
                lse2 = L > 0.f ? M + log2f(L) : -INFINITY;
                c_begin = 2 * b; c_end = min(2 * b + 2, D / 32);
            }
            const bool use0 = __any_sync(0xffffffffu, w0 != 0.f), use1 = __any_sync(0xffffffffu, w1 != 0.f);
            // A thread holds one row, but a row-per-thread store touches 32 lines per instruction: the
            // warp passes each 128-byte slice of its 32 rows through shared memory (its own rows of the Q
            // tile, which no MMA reads any more; 16-byte pieces XOR-swizzled by row) and writes whole lines.
            const int w4 = warp & 3;
            uint8_t* stage = smem + Geo::OFF_Q + b * (dual ? Geo::QTILE_BYTES : Geo::QHALF_BYTES) + w4 * 32 * 128;
            const int row_base = (dual ? 128 * b : 0) + 32 * w4;      // item row of the warp's first thread
            const bool final_out = it.partial_row0 < 0;
            auto flush = [&](int byte0) {      // byte0: offset of the slice inside an output row
                __syncwarp();
#pragma unroll (ALONE && D == 128 ? 4 : 8)
                for (int i = 0; i < 8; ++i) {
                    const int row = 4 * i + (lane >> 3), pc = lane & 7;
                    const uint4 v = *reinterpret_cast<const uint4*>(stage + row * 128 + ((pc ^ (row & 7)) << 4));
                    const int ri = row_base + row, tt = ri / G, gg = ri % G;
                    if (tt < it.ntok) {
                        uint8_t* dst = final_out
                            ? reinterpret_cast<uint8_t*>(out + ((size_t)(it.q_row0 + tt) * Hq + (size_t)it.kv_head * G + gg) * D)
                            : reinterpret_cast<uint8_t*>(p.partial_o + (((size_t)it.partial_row0 + tt) * G + gg) * D);
                        *reinterpret_cast<uint4*>(dst + byte0 + pc * 16) = v;
                    }
                }
                __syncwarp();
            };
#pragma unroll 1
            for (int c = c_begin; c < c_end; ++c) {
                float acc[32];
#pragma unroll
                for (int e = 0; e < 32; ++e) acc[e] = 0.f;
                if (use0) {
                    uint32_t ro[32];
                    tmem_ld32(lane_addr + kColO + 32u * c, ro);
                    tmem_wait_ld();
                    if (w0 != 0.f) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[e] = __uint_as_float(ro[e]) * w0;
                    }
                }
                if (use1) {
                    uint32_t ro[32];
                    tmem_ld32(lane_addr + kColO + (uint32_t)D + 32u * c, ro);
                    tmem_wait_ld();
                    if (w1 != 0.f) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[e] = fmaf(__uint_as_float(ro[e]), w1, acc[e]);
                    }
                }
                uint8_t* mine_row = stage + lane * 128;
                if (final_out) {
                    // 32 columns -> 64 bytes of bf16: pieces 4 (c & 1) .. + 3 of a 64-column slice
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        *reinterpret_cast<uint4*>(mine_row + ((((c & 1) * 4 + k) ^ (lane & 7)) << 4)) =
                            make_uint4(pack_bf16x2(acc[8 * k], acc[8 * k + 1]), pack_bf16x2(acc[8 * k + 2], acc[8 * k + 3]),
                                       pack_bf16x2(acc[8 * k + 4], acc[8 * k + 5]), pack_bf16x2(acc[8 * k + 6], acc[8 * k + 7]));
                    if (c & 1) flush((c >> 1) * 128);
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        *reinterpret_cast<uint4*>(mine_row + ((k ^ (lane & 7)) << 4)) =
                            make_uint4(__float_as_uint(acc[4 * k]), __float_as_uint(acc[4 * k + 1]),
                                       __float_as_uint(acc[4 * k + 2]), __float_as_uint(acc[4 * k + 3]));
                    flush(c * 128);
                }
            }
            if (row_valid && (dual || b == 0)) {
                if (it.partial_row0 < 0) {
                    if (lse != nullptr) lse[(size_t)(it.q_row0 + t) * Hq + hq] = lse2 * kLn2;
                } else {
                    p.partial_lse[prow * G + g] = lse2;
                }
            }
            tc_fence_before();
            mbar_arrive(bar(Geo::kOFree));
            if (lane == 0) trace_event(1 + warp, ev, 36);
            cnt += mine;
            kv_base += ntiles;
        }
        if ((threadIdx.x & 127) == 0) {
            trace_set(b ? 15 : 11, tr_wait);
            if (b == 0) { trace_set(12, tr_work); trace_set(13, tr_tiles); }
        }
    }

    // common exit: every role gets here, then the allocating warp releases tensor memory
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

}  // namespace tc

}  // namespace asynclm
