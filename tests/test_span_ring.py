"""Order of the span body's hand-offs (csrc/span_ring.h, csrc/attn_append_tc.cuh), on the CPU.

A barrier wait names only the parity of a phase: it tells phase k from phase k - 1, not from phase k - 2.
The model below builds, for a CTA's sequence of items, the order that the kernel's waits and program order
enforce among fills, arrivals, tensor-core turns, softmax steps and releases, with the slots and use counts taken
from the kernel's own header, and checks for every wait on a ring barrier that the phase before the one it
waits for is over whatever the warps' relative speed.  Tiles arrive in any order (their copies complete by
themselves); the MMA warps take turns, empty ones included, and those turns are part of the order.
"""
import ctypes
import os
import subprocess

import pytest

from paper_2412_07017_b200 import build as lib_build

PROBE = """
#include "span_ring.h"
using namespace asynclm::tc;
extern "C" int slots_of(int head_dim) { return ring_slots(head_dim); }
extern "C" int slot_of(int which, int t, int slots) { return ring_slot(which, t, slots); }
extern "C" int use_of(int t, int slots) { return ring_use(t, slots); }
extern "C" int carried(int t, int step, int n, int slots) {      // slot and parity of tile t + n * step, carried along from t
    RingPlace x = ring_place(t, slots);
    for (int k = 0; k < n; ++k) x = ring_next(x, step, slots);
    return 2 * x.slot + (int)x.parity;
}
extern "C" int by_rows(int kv_end, int last_tile, int page) { return last_page_by_rows(kv_end, last_tile != 0, page); }
"""


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, lib = os.path.join(d, "probe.cpp"), os.path.join(d, "probe.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", lib_build.CSRC, "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


def placed_by_kernel(ring, head_dim):
    """(kind, tile, its item's first tile, item's tiles, dual) -> (slot, uses of that slot before)"""
    n = ring.slots_of(head_dim)
    return lambda which, t, first, tiles, dual: (ring.slot_of(which, t, n), ring.use_of(t, n))


def placed_in_one_ring(slots):
    """K and V tiles in one ring in the order of consumption, restarted with every item: the mistake."""
    def place(which, t, first, tiles, dual):
        lead, g = 2 if dual else 4, t - first
        pos = 2 * first + (g + min(tiles, g + lead) if which else (g if g < lead else 2 * g - lead + 1))
        return pos % slots, pos // slots
    return place


def ambiguous_waits(items, place, turns=True):
    """items: (64-key tiles, dual) in the order a CTA runs them.  Returns the waits that could pass early.  Without
    `turns` the MMA warps issue as soon as their own waits are over."""
    before = {}          # node -> nodes known to come before it

    def after(node, *prev):
        before.setdefault(node, set()).update(p for p in prev if p is not None)
        return node

    waits = []           # (where the warp stands when it waits, what has to be over, description)
    used = {}            # slot -> {use: (kind, tile, groups that read it)}
    last = {}            # program order of each warp: its latest node
    turn_no = [0, 0]
    first, opened = 0, None
    for i, (n, dual) in enumerate(items):
        for t in range(first, first + n):
            for which in (0, 1):
                slot, use = place(which, t, first, n, dual)
                used.setdefault(slot, {})[use] = (which, t, (0, 1) if dual else ((t - first) & 1,))
        first += n
    first = 0
    for i, (n, dual) in enumerate(items):
        where = {(w, t): place(w, t, first, n, dual) for w in (0, 1) for t in range(first, first + n)}
        for which in (0, 1):                                   # producers: not tied to the items' ends
            for t in range(first, first + n):
                slot, use = where[which, t]
                here = last.get(("prod", which))
                if use >= 2:
                    w0, t0, groups = used[slot][use - 2]
                    waits += [(here, ("free", w0, t0, b), ("empty", which, t)) for b in groups]
                fill = after(("fill", which, t), here)
                if use >= 1:
                    w0, t0, groups = used[slot][use - 1]
                    after(fill, *[("free", w0, t0, b) for b in groups])
                last["prod", which] = fill
                after(("full", which, t), fill)
        ends = []
        for b in (0, 1):
            mine = [first + j for j in range(n) if dual or j % 2 == b]
            last["mma", b] = after(("open", i, b), last.get(("mma", b)), opened)
            last["soft", b] = after(("q", i, b), last.get(("soft", b)), opened)
            # group 0 has a tile more where they alternate and their number is odd: warp 1 makes up for it with an empty turn
            for u in range(-2, max(len(mine), (n + 1) // 2)):
                number, turn_no[b] = turn_no[b], turn_no[b] + 1
                turn = ("turn", b, number)
                if turns:      # turn k of warp 1 follows turn k of warp 0, turn k of warp 0 follows turn k - 1 of warp 1
                    after(turn, ("turn", 0, number) if b else ("turn", 1, number - 1) if number else None)
                if 0 <= u < len(mine):                         # softmax of tile u: its scores came with turn u - 2
                    s = after(("soft", i, b, u), last["soft", b], ("turn", b, number - 2))
                    after(("free", 0, mine[u], b), s)
                    if u >= 2:
                        after(("free", 1, mine[u - 2], b), s)
                    last["soft", b] = s
                    after(turn, s)
                reads = ([(1, mine[u])] if 0 <= u < len(mine) else []) + ([(0, mine[u + 2])] if u + 2 < len(mine) else [])
                here = last["mma", b]
                after(turn, here)
                for which, t in reads:
                    slot, use = where[which, t]
                    if use >= 1:
                        w0, t0, _ = used[slot][use - 1]
                        waits.append((here, ("full", w0, t0), ("full", which, t)))
                    after(turn, ("full", which, t))
                last["mma", b] = turn
            end = after(("end", i, b), last["soft", b], last["mma", b])
            for t in mine[-2:]:
                after(("free", 1, t, b), end)
            last["soft", b] = end
            ends.append(end)
        opened = after(("opened", i), *ends)
        first += n
    # ancestors as bit sets, in an order in which everything comes after what precedes it
    index, anc, stack = {}, {}, []
    for root in before:
        stack.append(root)
        while stack:
            node = stack[-1]
            todo = [p for p in before.get(node, ()) if p not in anc]
            if node in anc or not todo:
                stack.pop()
                if node not in anc:
                    index[node] = len(index)
                    bits = 1 << index[node]
                    for p in before.get(node, ()):
                        bits |= anc[p]
                    anc[node] = bits
            else:
                stack.extend(todo)
    return [what for here, need, what in waits if here is None or need not in index or not (anc[here] >> index[need]) & 1]


def three_items():
    for n1 in range(1, 13):
        for n2 in range(1, 13):
            for modes in range(8):
                yield [(n1, bool(modes & 1)), (n2, bool(modes & 2)), (12, bool(modes & 4))]


@pytest.mark.parametrize("head_dim", [128, 64])
def test_no_wait_on_a_ring_barrier_can_pass_a_phase_early(ring, head_dim):
    place = placed_by_kernel(ring, head_dim)
    for items in three_items():
        assert not ambiguous_waits(items, place), items
    assert not ambiguous_waits([(1, False)] * 30 + [(9, True), (2, False), (40, True)], place)


def test_the_model_finds_the_early_wait_of_a_shared_ring():
    """V5 of the first item frees a slot for the V producer while V0, two uses earlier, may be unread."""
    found = ambiguous_waits([(7, False), (1, False), (12, False)], placed_in_one_ring(10))
    assert any(kind == "empty" for kind, _, _ in found)
    assert not any(kind == "empty" for kind, _, _ in ambiguous_waits([(40, True)], placed_in_one_ring(10)))


def test_the_model_finds_the_early_waits_of_warps_that_take_no_turns(ring):
    """With five slots and alternating tiles, the tile a slot held before is the other group's: only the turns say that
    it has arrived."""
    found = ambiguous_waits([(12, False)], placed_by_kernel(ring, 128), turns=False)
    assert ("full", 0, 6) in found and ("full", 1, 6) in found
    assert not ambiguous_waits([(12, True)], placed_by_kernel(ring, 128), turns=False)


@pytest.mark.parametrize("head_dim", [128, 64])
def test_positions_carried_along_are_those_of_the_tiles(ring, head_dim):
    slots = ring.slots_of(head_dim)
    for first in range(3 * slots):
        for step in (1, 2):      # both groups on every tile, or alternate tiles
            for n in range(4 * slots):
                t = first + n * step
                assert ring.carried(first, step, n, slots) == 2 * ring.slot_of(0, t, slots) + ring.use_of(t, slots) % 2


def test_the_mma_warps_turns_are_as_modelled():
    """Each warp takes and passes its token once a turn, in empty turns and in the one that makes up for an odd tile, too."""
    with open(os.path.join(lib_build.CSRC, "attn_append_tc.cuh")) as f:
        role = f.read().split("MMA issuers", 1)[1].split("softmax / epilogue groups", 1)[0]
    turns, extra = role.split("for (int u = -2; u < mine && ok; ++u) {", 1)[1].split("if (!dual && b == 1 && (ntiles & 1) != 0) {", 1)
    empty, full = turns.split("if (!pv && !qk) {", 1)[1].split("continue;", 1)
    for part in (empty, extra):
        assert part.count("take_token(ok);") == 1 and part.count("pass_token();") == 1
    assert full.count("take_token(ok);") == 1
    assert full.index("wait_tile(1, ") < full.index("wait_tile(0, ") < full.index("take_token(ok);") < full.index("mma_f16")
    # passed among the MMAs of Q K^T, or behind the last MMA where there is none
    assert full.count("pass_token();") == 2 and "if (!qk) pass_token();" in full


def test_the_proxy_fence_stands_between_the_tiles_arrival_and_the_mmas_that_read_them(ring):
    """TMA copies and tcgen05.mma are both of the asynchronous proxy, but an unfinished last V page comes by cp.async,
    through the generic one: without a proxy fence behind the full barriers' waits nothing says that the MMAs see it.
    A missing fence need not show in any result, so what is checked is the order of the statements, and that one rule
    says which page comes that way and where the fence stands."""
    with open(os.path.join(lib_build.CSRC, "attn_append_tc.cuh")) as f:
        source = f.read()
    turn = source.split("for (int u = -2; u < mine && ok; ++u) {", 1)[1].split("mma_commit(el, done);", 1)[0]
    steps = ["wait_tile(1, ", "wait_tile(0, ", "fence_async_smem();", "mma_f16_ta(", "mma_f16("]
    at = [turn.index(s) for s in steps]
    assert at == sorted(at) and turn.count("fence_async_smem();") == 1 and "cp_async16(" not in turn
    assert "if (pv && last_page_by_rows(it.kv_end, j == ntiles - 1, kPage)) fence_async_smem();" in turn
    producer = source.split("producer warps\n", 1)[1].split("MMA issuers", 1)[0]
    assert "const bool ragged = which == 1 && last_page_by_rows(cur.kv_end, t == ntiles - 1, kPage);" in producer
    assert producer.count("cp_async16(") == 1 and "if (ragged) {" in producer.split("cp_async16(", 1)[0]
    for kv0 in (0, 64, 128, 4096):
        for kv_end in range(kv0 + 1, kv0 + 200):
            tiles = -(-(kv_end - kv0) // 64)
            for t in range(tiles):
                rows = min(64, kv_end - kv0 - 64 * t)
                assert bool(ring.by_rows(kv_end, t == tiles - 1, 16)) == (rows % 16 != 0)


@pytest.mark.parametrize("source,role,loop", [
    ("attn_append_tc.cuh", "producer warps\n", "for (int ii = i0; cur.kv_end > 0 && ok; ++ii) {"),
    ("attn_decode.cuh", "producer warp\n", "while (cur.kv_end > 0 && ok) {")])
def test_a_producer_stays_until_its_copies_have_landed(source, role, loop):
    """A copy that lands when its CTA's shared memory belongs to somebody else overwrites that.  A producer that is
    through cannot know that another role has given up, so the wait for the last copies depends on nothing."""
    with open(os.path.join(lib_build.CSRC, source)) as f:
        body = f.read().split(role, 1)[1].split(loop, 1)[1]
    depth, at = 1, 0
    while depth:
        depth += {"{": 1, "}": -1}.get(body[at], 0)
        at += 1
    rest = body[at:]
    drain = rest.index("land_copies(")
    depth = rest[:drain].count("{") - rest[:drain].count("}")
    assert depth == 0 and not rest[:drain].rstrip().endswith(("else", ")"))
