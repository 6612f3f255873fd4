// Where the span body's K and V tiles lie in shared memory, and the phases of the barriers that hand them
// over (device code; tests/test_span_ring.py compiles this file for the host).
//
// K tiles and V tiles have a ring each, filled by a producer warp each: tile t of the CTA (counted over all
// its items) is the t-th tile of its kind and takes slot t mod `slots`.  A barrier wait names only the parity
// of a phase, so a wait for phase k is sound only if phase k - 1 of the same barrier is known to be over:
//   empty (a producer waits before it fills tile t): the tile two uses earlier, t - 2 * slots, has been
//     released, because the same warp waited for that before it filled t - slots;
//   full (an MMA warp waits for tile t): tile t - slots has arrived.  It belongs to an item before (an item starts when
//     everything of the one before has been consumed), or the same MMA warp has waited for it, or, where the groups take
//     alternate tiles and `slots` is odd, the other one has: tiles arrive in any order (their copies complete by
//     themselves), and what says that the other warp has waited for that tile is that the warps take turns, each turn's
//     waits standing in front of its token.  With five slots the turns are a condition for these waits, not only
//     a matter of speed: tests/test_span_ring.py finds the early waits of warps without them.
// One ring for both kinds does not have the first property: a slot would pass from V to K and back to V
// without the V producer having waited for the tile in between, whose fill and release it does not see.
// Five slots each at head_dim 128 hold as many tiles, in the order of consumption, as one ring of ten (24 sequences
// with spans of up to 96 tokens, four layers: 399 us a pass with one ring, 390 with two; 32 layers of a mixed
// batch: 2284 and 2245-2275).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ASYNCLM_HD __host__ __device__
#else
#define ASYNCLM_HD
#endif

namespace asynclm {
namespace tc {

// Slots of one ring: 80 KiB of 64-key tiles.
ASYNCLM_HD constexpr int ring_slots(int head_dim) { return 640 / head_dim; }
// Slot (K ring first, then V ring) of the CTA's t-th K (which = 0) or V (which = 1) tile.
ASYNCLM_HD constexpr int ring_slot(int which, int t, int slots) { return which * slots + t % slots; }
// How often that slot has been used before.
ASYNCLM_HD constexpr int ring_use(int t, int slots) { return t / slots; }
// Where a tile lies in its ring and the parity of its phase, and the same `step` tiles further on (step <= slots), which
// costs the MMA warps less than the division.
struct RingPlace { int slot; uint32_t parity; };
ASYNCLM_HD constexpr RingPlace ring_place(int t, int slots) { return RingPlace{ring_slot(0, t, slots), (uint32_t)ring_use(t, slots) & 1u}; }
ASYNCLM_HD constexpr RingPlace ring_next(RingPlace x, int step, int slots) {
    x.slot += step;
    if (x.slot >= slots) { x.slot -= slots; x.parity ^= 1u; }
    return x;
}
// Whether an item's last tile has a last page that is not full (`page`: a power of two; items begin on a page boundary).
// V's is copied row by row through the generic proxy, with zeros behind the end, and the MMAs that read it need a proxy fence.
ASYNCLM_HD constexpr bool last_page_by_rows(int kv_end, bool last_tile, int page) { return last_tile && (kv_end & (page - 1)) != 0; }

}  // namespace tc
}  // namespace asynclm
