"""Plans of middling size are uploaded by a kernel out of a page-locked workspace, and the kernels behind read them ahead of
their wait for the one in front: whatever comes first behind an upload sees that plan and no older one."""
import ctypes

import numpy as np
import pytest

from paper_2412_07017_b200 import binding as B
from paper_2412_07017_b200 import workload as W

pytestmark = pytest.mark.gpu
SHAPE = W.Shape(32, 8, 64, 16)


class Batch:
    """24 sequences in one pool; the same lengths with another page table each time, so that plans differ in page ids only."""

    def __init__(self):
        import torch
        g = np.random.default_rng(5)
        self.ctx = g.integers(200, 900, 24).astype(np.int32)
        self.qi = np.arange(25, dtype=np.int32)
        need = -(-(self.ctx + 1) // 16)
        self.pi = np.zeros(25, np.int32)
        self.pi[1:] = np.cumsum(need)
        self.pages = int(self.pi[-1]) + 300
        torch.manual_seed(1)
        self.pool = torch.randn(self.pages, 2, 8, 16, 64, device="cuda").bfloat16()
        self.q = torch.randn(24, 32, 64, device="cuda").bfloat16()
        self.k, self.v = (torch.randn(24, 8, 64, device="cuda").bfloat16() for _ in range(2))
        host, dev = B.workspace_size(SHAPE, self.pages, 24, 24, int(self.pi[-1]))
        self.dev_ws = torch.empty(dev, dtype=torch.uint8, device="cuda")
        self.host_bytes = host
        torch.cuda.synchronize()

    def ids(self, k):
        return np.random.default_rng(100 + k).permutation(self.pages)[:self.pi[-1]].astype(np.int32)

    def plan(self, ids, host_ws):
        return B.asynclm_plan(SHAPE, self.pages, self.qi, self.ctx, self.pi, ids, host_ws=host_ws, dev_ws=self.dev_ws)

    def pinned(self):
        import torch
        return torch.empty(self.host_bytes, dtype=torch.uint8).pin_memory()

    def call(self, plan, kind, pool, out):
        if kind == "step":
            B.asynclm_step(plan, self.q, self.k, self.v, pool, out, None)
        else:
            if kind == "rope":
                B.asynclm_kv_append_rope(plan, self.k, self.v, pool, None, 1e4)
            elif kind == "calls":
                B.asynclm_kv_append(plan, self.k, self.v, pool)
            (B.asynclm_attn_mixed_static if kind == "static" else B.asynclm_attn_mixed)(plan, self.q, pool, out, None)


def bits(x):
    import torch
    return x.view(torch.int16).cpu()


def blob_bytes(plan):
    """Bytes of the plan itself: the device workspace without the partial rows behind it."""
    rows, a256 = plan.info["partial_rows"] * SHAPE.num_q_heads // SHAPE.num_kv_heads, lambda x: -(-x // 256) * 256
    return plan.info["device_bytes_used"] - a256(rows * SHAPE.head_dim * 4) - a256(rows * 4)


KERNEL, COPY = 0, 1      # of CUgraphNodeType


def nodes_of(call):
    """What `call(stream)` enqueues: the types of the nodes that it leaves in a capture."""
    import torch
    cu, s, graph, n = ctypes.CDLL("libcuda.so.1"), torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_size_t()
    raw = ctypes.c_void_p(s.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(raw, 2) == 0      # (relaxed: the mode does not matter to what is called here)
    try:
        call(s)
    finally:
        assert cu.cuStreamEndCapture(raw, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes, kind = (ctypes.c_void_p * n.value)(), ctypes.c_int()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    assert cu.cuGraphDestroy(graph) == 0
    return kinds


@pytest.mark.parametrize("want", [32768 - 256, 32768, 32768 + 4096, 300 << 10, (600 << 10) + 256, (1 << 20) + 512, (2 << 20) - 256, 2 << 20, (2 << 20) + 256])
def test_plans_of_middling_size_go_by_kernel_and_arrive_whole(want):
    """Plans of `want` bytes, by page table entries that no key needs yet (4 bytes each, sections of 256)."""
    import torch
    t = Batch()
    few = 4 if want < 65536 else 24      # sequences (24 have a plan of 83 712 bytes at least)
    qi, ctx, pi = t.qi[:few + 1], t.ctx[:few], t.pi[:few + 1].copy()
    ids = t.ids(0)
    dry = lambda n: B.plan_host(SHAPE, t.pages, qi, ctx, np.append(pi[:-1], n).astype(np.int32), np.resize(ids, n))
    at = int(pi[-1]) + (want - blob_bytes(dry(int(pi[-1])))) // 4
    pi[-1] = at
    ids = np.resize(ids, at)
    host, dev = B.workspace_size(SHAPE, t.pages, few, few, at)
    dev_ws = torch.full((dev,), 0xA5, dtype=torch.uint8, device="cuda")
    ws = torch.zeros(host, dtype=torch.uint8).pin_memory()
    plan_of = lambda s=None: B.asynclm_plan(SHAPE, t.pages, qi, ctx, pi, ids, stream=s, host_ws=ws, dev_ws=dev_ws)
    torch.cuda.synchronize()
    assert nodes_of(plan_of) == [KERNEL if 32768 <= want <= 2 << 20 else COPY]
    assert (dev_ws == 0xA5).all()
    plan = plan_of()
    torch.cuda.synchronize()
    assert blob_bytes(plan) == want
    start = plan.info["host_bytes_used"] - want - -(-plan.info["num_items"] // 64) * 256      # behind the plan: the CTA of each item
    assert torch.equal(dev_ws[:want].cpu(), ws[start:start + want]) and (dev_ws[want:] == 0xA5).all()


@pytest.mark.parametrize("kind", ["calls", "step", "rope", "attention", "static"])
def test_steps_in_a_row_see_their_own_plan(kind):
    """One device workspace, planned anew ahead of every step without waiting for anything, page-locked against pageable memory
    (a copy in the stream) with a synchronisation around every call."""
    import torch
    t = Batch()
    want = []
    for k in range(6):
        pool, out = t.pool.clone(), torch.empty_like(t.q)
        plan = t.plan(t.ids(k), torch.empty(t.host_bytes, dtype=torch.uint8))
        assert blob_bytes(plan) >= 32768      # by kernel, from page-locked memory
        torch.cuda.synchronize()
        t.call(plan, kind, pool, out)
        torch.cuda.synchronize()
        want.append((bits(pool), bits(out)))
    pools, outs = [t.pool.clone() for _ in range(6)], [torch.empty_like(t.q) for _ in range(6)]
    slots, ids = [t.pinned() for _ in range(6)], [t.ids(k) for k in range(6)]
    torch.cuda.synchronize()
    for k in range(6):
        plan = t.plan(ids[k], slots[k])
        for _ in range(2):
            t.call(plan, kind, pools[k], outs[k])
    torch.cuda.synchronize()
    assert B.last_device_status(plan) == 0
    for k in range(6):
        assert torch.equal(bits(pools[k]), want[k][0]) and torch.equal(bits(outs[k]), want[k][1]), k


def test_captured_launches_and_launches_behind_a_capture():
    """A capture between the upload and the first launch leaves that launch the first; the graph, replayed behind later uploads into the
    same workspace, sees the plan that is there."""
    import torch
    t = Batch()
    ws = [t.pinned() for _ in range(3)]
    out = torch.empty_like(t.q)
    warm = t.plan(t.ids(0), ws[0])
    t.call(warm, "calls", t.pool.clone(), out)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    pool, pool2 = t.pool.clone(), t.pool.clone()
    out2 = torch.empty_like(t.q)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        plan = t.plan(t.ids(1), ws[1])
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            t.call(plan, "calls", pool, out)
            t.call(plan, "calls", pool, out)
        t.call(plan, "calls", pool2, out2)
        g.replay()
        s.synchronize()
        assert torch.equal(bits(out), bits(out2)) and torch.equal(bits(pool), bits(pool2))
        first = bits(out)
        t.plan(t.ids(2), ws[2])
        g.replay()
        s.synchronize()
        again, ref = bits(out), torch.empty_like(t.q)
        plan = t.plan(t.ids(2), torch.empty(t.host_bytes, dtype=torch.uint8))
        s.synchronize()
        t.call(plan, "attention", pool, ref)
        s.synchronize()
    assert torch.equal(again, bits(ref)) and not torch.equal(again, first)


def test_a_workspace_of_two_registrations_is_refused():
    """Page-locked in two parts that no single range covers: the copy refuses it, and no kernel reads it."""
    import torch
    t = Batch()
    cut, base = 32768, torch.empty(t.host_bytes + 8192, dtype=torch.uint8)
    base, rt = base[-base.data_ptr() % 4096:], torch.cuda.cudart()
    parts = [(base.data_ptr(), cut), (base.data_ptr() + cut, -(-(t.host_bytes - cut) // 4096) * 4096)]
    t.dev_ws.zero_()
    for p, n in parts:
        assert int(rt.cudaHostRegister(p, n, 0)) == 0
    try:
        with pytest.raises(B.AsynclmError, match="CUDA"):
            t.plan(t.ids(1), base[:t.host_bytes])
        torch.cuda.synchronize()
    finally:
        for p, n in parts:
            rt.cudaHostUnregister(p)
    assert not t.dev_ws.any()


def test_a_captured_upload():
    """The upload itself in a graph reads what the host workspace holds when the graph is launched."""
    import torch
    t = Batch()
    ws, out, ref = t.pinned(), torch.empty_like(t.q), torch.empty_like(t.q)
    pool = t.pool.clone()
    t.call(t.plan(t.ids(0), ws), "calls", pool, out)
    torch.cuda.synchronize()
    s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            plan = t.plan(t.ids(1), ws)
            t.call(plan, "calls", pool, out)
            t.call(plan, "attention", pool, out)
        for k in (1, 2):
            if k == 2:      # another plan of the same lengths, written by the planner on the host only
                keep = ws.clone()
                t.plan(t.ids(2), ws)
                s.synchronize()
                assert not torch.equal(keep, ws)
                t.dev_ws.zero_()
            g.replay()
            s.synchronize()
            t.call(t.plan(t.ids(k), torch.empty(t.host_bytes, dtype=torch.uint8)), "attention", pool, ref)
            s.synchronize()
            assert torch.equal(bits(out), bits(ref)), k
