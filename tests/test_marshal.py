"""The binding's marshalling: what a function at the other end is given for every kind of argument, and what is refused."""
import ctypes as C

import pytest
import torch

import paper_2507_07114_b200 as L
from paper_2507_07114_b200 import binding


@pytest.fixture(scope="module")
def call():
    L.load_library()
    return binding._native


def receiver(n, rc=0, tables=()):
    """A C function of n 64-bit arguments; what it got, with the first 64 entries of the tables among them."""
    got = []

    def f(*a):
        got.append([[C.cast(x, C.POINTER(C.c_uint64))[i] for i in range(64)] if k in tables else x for k, x in enumerate(a)])
        return rc

    fn = C.CFUNCTYPE(C.c_int, *[C.c_uint64] * n)(f)
    return fn, C.cast(fn, C.c_void_p).value, got


class Named(torch.Tensor):
    pass


class Elsewhere:
    def data_ptr(self):
        return 0x1230


def test_arguments_arrive(call):
    a, b = torch.zeros(8), torch.nn.Parameter(torch.ones(4, dtype=torch.bfloat16))
    sub = torch.zeros(3).as_subclass(Named)
    rows = torch.zeros(3, 16)
    fn, at, got = receiver(9, rc=7, tables=(2, 5, 8))
    made = bytes(range(1, 9)) * 64
    rc = call(at, "utpptpub", C.c_void_p(0xABC0), 2 ** 64 + 5, [a, None, b, sub, Elsewhere()], a[2:], None, rows, b, -1, made)
    assert rc == 7
    g = got[0]
    assert g[0] == 0xABC0 and g[1] == 5                                        # integers modulo 2^64, as ctypes takes them
    assert g[2] == [a.data_ptr(), 0, b.data_ptr(), sub.data_ptr(), 0x1230] + [0] * 59
    assert g[3] == a.data_ptr() + 8 and g[4] == 0
    assert g[5] == [rows[i].data_ptr() for i in range(3)] + [0] * 61            # a stacked tensor is a sequence of its rows
    assert g[6] == b.data_ptr() and g[7] == 2 ** 64 - 1 and g[8] == [int.from_bytes(made[:8], "little")] * 64


def test_long_tables_and_every_count_of_arguments(call):
    ts = tuple(torch.zeros(1) for _ in range(100))
    fn, at, got = receiver(2, tables=(1,))
    assert call(at, "t", None, ts) == 0
    assert got[0] == [0, [t.data_ptr() for t in ts[:64]]]
    for n in range(1, 17):
        fn, at, got = receiver(n, rc=n)
        assert call(at, "u" * (n - 1), 9, *range(1, n)) == n and got[0] == [9, *range(1, n)]


def test_refusals(call):
    fn, at, got = receiver(2)
    for args in [(at, "u", None, 1.5), (at, "u", None, None), (at, "p", None, 3), (at, "t", None, 3), (at, "t", None, [3]), (at, "u", None),
                 (at, "u", None, 1, 2), (at, "b", None, "text"), (at, "u", "text", 1), (0, "u", None, 1), (at, "u" * 16, None, *[1] * 16), (at,)]:
        with pytest.raises((TypeError, ValueError, AttributeError)):
            call(*args)
    with pytest.raises(RuntimeError):                                           # no storage: torch's own exception, not an abort
        torch.func.vmap(lambda t: call(at, "p", None, t) or t)(torch.zeros(2, 2))
    assert got == []


@pytest.mark.gpu
def test_an_error_of_the_library_is_raised():
    with pytest.raises(L.LossyError) as e:
        L.lossy_step(None, 1, None, None, None)
    assert e.value.code == binding.LOSSY_EINVAL
