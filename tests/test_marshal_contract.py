"""What the calls of the binding take and refuse is what ctypes takes and refuses for the library's signatures, whichever way the
arguments go."""
import ctypes as C
import struct
from types import SimpleNamespace

import pytest
import torch

from paper_2507_07114_b200 import binding


@pytest.fixture
def received(monkeypatch):
    """A library whose lossy_step and lossy_packet_sqnorms note their arguments; no stream, so that no device is asked."""
    binding.load_library()
    got = []

    def note(name, argtypes, kinds, tables):
        def f(*a):
            got.append([C.cast(x, C.POINTER(C.c_uint64))[:2] if k in tables else x for k, x in enumerate(a)])
            return 0
        keep.append(C.CFUNCTYPE(C.c_int, *[C.c_uint64] * len(argtypes))(f))
        address = C.cast(keep[-1], C.c_void_p).value
        fn = C.CFUNCTYPE(C.c_int, *argtypes)(address)
        monkeypatch.setitem(binding._NATIVE, name, kinds)
        setattr(lib, name, fn)
        lib.at[name] = address

    keep, lib = [], SimpleNamespace(at={})
    vp, u64 = C.c_void_p, C.c_uint64
    note("lossy_step", [vp, u64] + [vp] * 5, "uppppp", ())
    note("lossy_packet_sqnorms", [vp] * 3, "tp", (1,))
    note("lossy_fused_step", [vp, u64] + [vp] * 12, "utppptpppppps", (2, 6))
    monkeypatch.setattr(binding, "load_library", lambda: lib)
    return got


class Whole:
    _as_parameter_ = 7


class Pointer:
    def __init__(self, at):
        self.at = at

    def data_ptr(self):
        return self.at


def test_integers_and_contexts_as_ctypes_takes_them(received):
    t = torch.zeros(8)
    for step, want in ((5, 5), (True, 1), (-1, 2 ** 64 - 1), (C.c_uint64(9), 9), (Whole(), 7)):
        binding.lossy_step(None, step, t, None, t)
        assert received[-1] == [0, want, t.data_ptr(), 0, t.data_ptr(), 0, 0]
    held = C.c_uint64(3)
    for ctx, want in ((C.c_void_p(64), 64), (C.c_void_p(), 0), (128, 128), (C.pointer(held), C.addressof(held)), (C.byref(held), C.addressof(held))):
        binding.lossy_step(ctx, 1, t, None, t)
        assert received[-1][0] == want
    binding.lossy_step(None, 1, Pointer(None), None, Pointer(-16))
    assert received[-1] == [0, 1, 0, 0, 2 ** 64 - 16, 0, 0]
    binding.lossy_packet_sqnorms(None, {t: 0, None: 1}, t)                   # anything with a length that can be walked
    assert received[-1] == [0, [t.data_ptr(), 0], t.data_ptr()]


def test_refusals_as_ctypes_refuses(received):
    t = torch.zeros(8)
    for step in (1.5, None, "1", C.c_int32(1), C.c_uint32(1)):
        with pytest.raises(C.ArgumentError):
            binding.lossy_step(None, step, t, None, t)
    for ctx in (C.c_uint64(64), C.c_int32(64), 1.5, SimpleNamespace(value=64)):      # an integer object is no address
        with pytest.raises(C.ArgumentError):
            binding.lossy_step(ctx, 1, t, None, t)
    for table in ((x for x in (t, t)), 3):
        with pytest.raises(TypeError):
            binding.lossy_packet_sqnorms(None, table, t)
    with pytest.raises(AttributeError):
        binding.lossy_step(None, 1, 3, None, t)
    with pytest.raises(struct.error):
        binding.lossy_packet_sqnorms(None, [Pointer(-16)], t)
    assert received == []


def test_a_prepared_step_takes_the_same_integers(received):
    t = torch.zeros(8)
    call = binding.lossy_fused_step_prepared(None, [t, t], t, None, None, [t, t], stream=SimpleNamespace(cuda_stream=48))
    for step, want in ((5, 5), (C.c_uint64(9), 9), (Whole(), 7)):
        call(step)
        assert received[-1][:4] == [0, want, [t.data_ptr()] * 2, t.data_ptr()] and received[-1][-1] == 48
    with pytest.raises(C.ArgumentError):
        call(1.5)
