// Where the span body's K and V tiles lie in shared memory, and the phases of the barriers that hand them
// over (device code; tests/test_span_ring.py compiles this file for the host).
//
// K tiles and V tiles have a ring each, filled by a producer warp each: tile t of the CTA (counted over all
// its items) is the t-th tile of its kind and takes slot t mod `slots`.  A barrier wait names only the parity
// of a phase, so a wait for phase k is sound only if phase k - 1 of the same barrier is known to be over:
//   empty (a producer waits before it fills tile t): the tile two uses earlier, t - 2 * slots, has been
//     released, because the same warp waited for that before it filled t - slots;
//   full (an MMA warp waits for tile t): tile t - slots has been filled, because it belongs to an item
//     before (an item starts when everything of the one before has been consumed) or was filled, in
//     order, ahead of a tile of this item that the same MMA warp has waited for.
// One ring for both kinds does not have the first property: a slot would pass from V to K and back to V
// without the V producer having waited for the tile in between, whose fill and release it does not see.
// Five slots each at head_dim 128 hold as many tiles, in the order of consumption, as one ring of ten (24 sequences
// with spans of up to 96 tokens, four layers: 399 us a pass with one ring, 390 with two; 32 layers of a mixed
// batch: 2284 and 2245-2275).
#pragma once

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

}  // namespace tc
}  // namespace asynclm
