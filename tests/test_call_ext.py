"""The extension that marshals the per-layer calls takes what needs no conversion and leaves the rest to ctypes; both ways
lead to the same call."""
import array
import os
import types
import warnings

import numpy as np
import pytest

from paper_2412_07017_b200 import binding as B
from paper_2412_07017_b200 import build as lib_build
from paper_2412_07017_b200 import workload as W


def fake(ptr, n=0):
    return types.SimpleNamespace(data_ptr=lambda: ptr, numel=lambda: n)


def ext():
    if lib_build.build_call_ext() is None:
        pytest.skip("no C compiler or Python header here: the calls go through ctypes")
    e = B._calls()
    assert e, "it was built, but cannot be loaded or bound"
    return e


STREAM = types.SimpleNamespace(cuda_stream=0)
I32 = np.array([0, 1], np.int32)


@pytest.mark.parametrize("a,taken", [
    (I32, True), (array.array("i", [0, 1]), True), (np.array([0, 1, 5], np.int32)[:2], True),
    ([0, 1], False), (np.array([0, 1]), False), (np.array([0, 9, 1, 9], np.int32)[::2], False), (I32.reshape(1, 2), False),
    (I32.astype(">i4"), False), (I32.astype(np.uint32), False), (I32.astype(np.float32), False)])
@pytest.mark.parametrize("at", range(4))
def test_only_arrays_that_need_no_conversion_are_taken(a, taken, at):
    arrays = [I32, I32[:1], I32, I32]
    arrays[at] = a
    # (a host workspace that is not 16-byte aligned: the call itself ends on its first checks)
    got = ext().plan(W.Shape(8, 2, 64, 16), 4, *arrays, STREAM, 0.0, fake(8, 8), fake(256, 8))
    assert (got is not None) == taken
    if taken:
        assert got[0] == -1 and got[1] == 0


def test_what_is_refused_is_refused_with_the_same_exceptions():
    e = ext()
    assert e.plan(W.Shape(8, 2, "64", 16), 4, I32, I32[:1], I32, I32, STREAM, 0.0, fake(8, 8), fake(256, 8)) is None
    with pytest.raises(AttributeError):
        e.append(0, None, fake(16), fake(16), STREAM)      # only `lse` and `q_inout` may be None
    with pytest.raises(AttributeError):
        e.attn(0, fake(16), fake(16), fake(16), None, object())
    with pytest.raises(TypeError):
        e.step(0)
    for rc in (e.append(0, fake(16), fake(16), fake(16), STREAM), e.append_rope(0, fake(16), fake(16), fake(16), None, 1e4, STREAM),
               e.attn(0, fake(16), fake(16), fake(16), None, STREAM), e.step(0, *[fake(16)] * 5, None, STREAM)):
        assert rc == -1      # no plan


def test_an_extension_that_fails_is_named_and_an_old_one_is_not_used(monkeypatch, tmp_path):
    def broken(force=False):
        raise RuntimeError("cc failed: no such struct")
    with monkeypatch.context() as m:
        m.setattr(B, "_call_ext", None)
        m.setattr(lib_build, "build_call_ext", broken)
        with pytest.warns(RuntimeWarning, match="no such struct"):
            assert B._calls() is False
        assert B._calls() is False      # once is enough
    with monkeypatch.context() as m:      # nothing to build it with, and none or an old one there
        old = tmp_path / "call_ext.so"
        m.setattr(lib_build, "CALL_EXT", str(old))
        m.setattr(lib_build.shutil, "which", lambda name: None)
        m.setattr(B, "_call_ext", None)
        assert lib_build.build_call_ext() is None
        old.write_bytes(b"")
        os.utime(old, (1, 1))
        assert lib_build.build_call_ext() is None
        with warnings.catch_warnings():
            warnings.simplefilter("error")
            assert B._calls() is False


def test_a_small_plan_holds_headers_of_the_ctas_it_uses_only():
    p = B.plan_host(W.Shape(8, 2, 64, 16), 40, [0, 1, 2], [100, 200], [0, 7, 20], list(range(20)))
    used = int(p.items()["cta"].max()) + 1
    assert 0 < used < 148 and 384 * used <= p.info["device_bytes_used"] < 384 * 148
    assert p.info["num_ctas_cuda"] == p.info["num_ctas_tensor"] == used
    n = 300      # sequences whose work is queued: every CTA takes part
    p = B.plan_host(W.Shape(8, 2, 64, 16), 20 * n, list(range(n + 1)), [300] * n, [20 * k for k in range(n + 1)], list(range(20 * n)))
    assert (p.items()["cta"] < 0).any() and p.info["num_ctas_cuda"] == 148


@pytest.mark.gpu
@pytest.mark.parametrize("side_stream", [False, True])
def test_both_ways_make_the_same_calls(monkeypatch, side_stream):
    import torch
    shape = W.Shape(8, 2, 64, 16)
    wl = W.make_single_step("ext", shape, [300, 40, 129], [1, 20, 1], seed=3)
    st = wl.steps[0]
    host, dev = B.workspace_size(shape, wl.num_pages, 3, 22, len(st.page_indices))
    results = []
    for way in (ext(), False):
        monkeypatch.setattr(B, "_call_ext", way)
        pool, q, k, v = (torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (wl.kv_pool, st.q, st.k_new, st.v_new))
        out, lse = torch.zeros_like(q), torch.zeros(q.shape[:2], dtype=torch.float32, device="cuda")
        out2 = torch.zeros_like(q)
        torch.cuda.synchronize()
        s = torch.cuda.Stream() if side_stream else None
        ws = torch.empty(host, dtype=torch.uint8).pin_memory(), torch.empty(dev, dtype=torch.uint8, device="cuda")
        plan = B.asynclm_plan(shape, wl.num_pages, *(np.asarray(x, np.int32) for x in (st.q_indptr, st.kv_len_before, st.page_indptr, st.page_indices)),
                              stream=s, host_ws=ws[0], dev_ws=ws[1])
        B.asynclm_kv_append_rope(plan, k, v, pool, q, 1e4, stream=s)
        B.asynclm_kv_append(plan, k, v, pool, stream=s)
        B.asynclm_attn_mixed(plan, q, pool, out, lse, stream=s)
        B.asynclm_step(plan, q, k, v, pool, out2, None, stream=s)
        torch.cuda.synchronize()
        assert B.last_device_status(plan) == 0
        with pytest.raises(B.AsynclmError):
            B.asynclm_plan(shape, 1, st.q_indptr.astype(np.int32), st.kv_len_before.astype(np.int32), st.page_indptr.astype(np.int32),
                           st.page_indices.astype(np.int32), host_ws=ws[0], dev_ws=ws[1])
        results.append([x.view(torch.int16).cpu() if x.dtype == torch.bfloat16 else x.cpu() for x in (pool, q, out, lse, out2)])
    assert all(torch.equal(a, b) for a, b in zip(*results))
