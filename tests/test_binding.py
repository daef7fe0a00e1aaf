"""Host side of the Python binding: the packed job list of the grouped calls has the
layout of the ctypes structure that is checked against the C header, and the
stream of a call without one (no GPU)."""
import ctypes
import sys
import types

import paper_0808_0487_gb300 as dwt


class _Plan:
    handle = 0x1122334455667788


def test_job_list_has_the_structure_s_layout():
    rows = [(_Plan, 0x0102030405060708, 0x1112131415161718, -5, 1 << 40, -(1 << 41)), (_Plan, None, 7, 2, 3, 4)]
    buf = dwt._jobs(rows)
    assert len(buf) == 2 * ctypes.sizeof(dwt._Job)
    for i, r in enumerate(rows):
        j = dwt._Job.from_buffer_copy(buf, i * ctypes.sizeof(dwt._Job))
        assert (j.plan, j.in_, j.out, j.batch, j.ld_in, j.ld_out) == (r[0].handle,) + r[1:]


def test_packing_follows_the_structure():
    # a structure of other order and padding: the format comes from it, not from a copy
    class Other(ctypes.Structure):
        _fields_ = [("a", ctypes.c_int), ("b", ctypes.c_longlong), ("c", ctypes.c_int), ("d", ctypes.c_void_p), ("e", ctypes.c_int)]

    x = Other.from_buffer_copy(dwt._packer(Other).pack(1, -2, 3, 4, -5))
    assert (x.a, x.b, x.c, x.d, x.e) == (1, -2, 3, 4, -5)
    assert dwt._packer(dwt._Job).format == dwt._JOB.format


def _torch(raw):
    t = types.ModuleType("torch")
    t.cuda = types.SimpleNamespace(is_initialized=lambda: True, is_available=lambda: True,
                                   current_stream=lambda: types.SimpleNamespace(cuda_stream=42))
    t._C = types.SimpleNamespace(**raw)
    return t


def test_stream_without_torch_s_raw_handle(monkeypatch):
    monkeypatch.setitem(sys.modules, "torch", _torch({"_cuda_getDevice": lambda: 1, "_cuda_getCurrentRawStream": lambda d: 70 + d}))
    assert dwt._stream(None) == 71
    for raw in ({}, {"_cuda_getDevice": lambda: 0}):   # a torch release without them
        monkeypatch.setitem(sys.modules, "torch", _torch(raw))
        assert dwt._stream(None) == 42
    assert dwt._stream(5) == 5
