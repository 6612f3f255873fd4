"""The C ABI library loads and exports every function include/asynclm.h declares (no GPU calls)."""
import ctypes
import os
import re

from paper_2412_07017_b200 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "asynclm.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(asynclm_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_function_is_exported():
    lib = B.load()
    names = declared_functions()
    assert len(names) >= 10
    for n in names:
        assert hasattr(lib, n), n
    assert set(B.EXPORTS) == set(names)


def test_version_and_strerror():
    lib = B.load()
    assert lib.asynclm_version() >= 100
    assert B.strerror(0) == "ok"
    for code in range(-8, 0):
        assert B.strerror(code) not in ("ok", "unknown status")
    assert B.strerror(-99) == "unknown status"


def test_struct_sizes_match_header_layout():
    assert ctypes.sizeof(B.CShape) == 32
    assert ctypes.sizeof(B.CPlanOptions) == 16
    assert ctypes.sizeof(B.CPlanInfo) == 12 * 4 + 3 * 8
    assert B.ITEM_DTYPE.itemsize == 32


def test_stream_handles_do_not_depend_on_a_private_function_of_torch(monkeypatch):
    import types

    import torch
    stream = types.SimpleNamespace(cuda_stream=0x5550)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: stream)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 0x7000 + device, raising=False)
    assert B._stream_ptr(None) == 0x7003
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert B._stream_ptr(None) == 0x5550
    assert B._stream_ptr(types.SimpleNamespace(cuda_stream=7)) == 7
