"""Calls through the C marshalling module take what the ctypes declarations take, and pass on the same numbers."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2510_22556_b200 import binding as B
from paper_2510_22556_b200.build import build_test_hooks

fastcall = pytest.importorskip("paper_2510_22556_b200._fastcall")


@pytest.fixture(scope="module")
def chunk():
    """An entry point of the test build that only computes: (parameter block, layers, sequences, offsets, longest, rows)."""
    l = C.CDLL(build_test_hooks())
    return fastcall.bind(C.cast(l.sablock_test_host_chunk, C.c_void_p).value)


@pytest.fixture(scope="module")
def block():
    return B.make_params(32, 8, 128, 32, torch.bfloat16)


@pytest.mark.parametrize("layers", [9, np.int64(9), np.int32(9), np.uint8(9), torch.tensor(9), 9 + (1 << 32)])
def test_scalars(chunk, block, layers):
    assert chunk(C.addressof(block), layers, 1, (0, 2100), np.int64(2100), 64) == 2


@pytest.mark.parametrize("cu", [(0, 2100), [0, 2100], [0.0, 2100.0], ["0", "2100"], list(np.array([0, 2100])), list(torch.tensor([0, 2100])),
                                [0, 2100 + (1 << 32)], [0, 2100] + [7] * 300])
def test_sequences(chunk, block, cu):
    assert chunk(C.addressof(block), 9, 1, cu, 2100, 64) == 2


def test_sequences_from_other_containers(chunk, block):
    for cu in (np.array([0, 2100]), torch.tensor([0, 2100]), range(0, 2101, 2100)):
        assert chunk(C.addressof(block), 9, 1, B._iarr(cu), 2100, 64) == 2


def test_none_is_a_null_pointer(chunk):
    assert B.lib().compress(None, None, None, None, None, 4096, 256, (1, 2), 2, None, None, None, None, None, 0, None) == 1


@pytest.mark.parametrize("bad", [1.5, "9", object()])
def test_what_is_no_integer_is_refused(chunk, block, bad):
    with pytest.raises(TypeError):
        chunk(C.addressof(block), bad, 1, (0, 2100), 2100, 64)
    with pytest.raises((TypeError, ValueError)):
        chunk(C.addressof(block), 9, 1, (0, object()), 2100, 64)


def test_a_list_that_changes_while_it_is_read(chunk, block):
    class Shrinks:
        def __init__(self, xs):
            self.xs = xs

        def __int__(self):
            self.xs.clear()
            return 0

    xs = []
    xs += [Shrinks(xs), 2100]
    assert chunk(C.addressof(block), 9, 1, xs, 2100, 64) == 2


def test_the_binding_takes_numpy_integers():
    p = B.make_params(32, 8, 128, 32, torch.bfloat16)
    fake = torch.zeros(4, dtype=torch.uint8)
    with pytest.raises(B.SablockError) as err:                   # refused for its workspace, not for the type of its budget
        B._check(B.lib().compress(C.addressof(p), fake.data_ptr(), fake.data_ptr(), fake.data_ptr(), fake.data_ptr(), 4096, np.int64(256),
                                  [np.int64(1), np.int64(2)], 2, fake.data_ptr(), fake.data_ptr(), fake.data_ptr(), fake.data_ptr(),
                                  fake.data_ptr(), 4, None), "sablock_compress")
    assert err.value.code == 3


def test_a_decoding_step_passes_what_the_tensors_say():
    """(on the CPU: a callback in the entry point's place, tensors that are views and carry an offset)"""
    seen = []
    proto = C.CFUNCTYPE(C.c_int, *[C.c_uint64] * 12)
    fn = proto(lambda *a: seen.append(a) or 7)
    step = fastcall.bind_decode(C.cast(fn, C.c_void_p).value)
    q = torch.zeros(5, 4, 8)[1:4]
    k, v = torch.zeros(3, 2, 11, 2, 8).unbind(1)
    out, ws, n = torch.zeros(3, 4, 8), torch.zeros(300, dtype=torch.uint8)[44:], torch.zeros(3, dtype=torch.int32)
    assert step(np.int64(99), q, k, v, n, out, None, ws, 1 << 40) == 7
    assert seen == [(99, 3, q.data_ptr(), k.data_ptr(), v.data_ptr(), 11, n.data_ptr(), out.data_ptr(), 0, ws.data_ptr(), 256, 1 << 40)]
    with pytest.raises(ValueError):
        step(99, q[0], k, v, None, out, None, ws, 0)
    with pytest.raises(IndexError):
        step(99, q, k[0, :, 0, 0], v, None, out, None, ws, 0)
    with pytest.raises(AttributeError):
        step(99, q, k, 5, None, out, None, ws, 0)
    with pytest.raises(TypeError):
        step(99, q, k, v, None, out, None, ws)
    with pytest.raises(TypeError):
        step(9.5, q, k, v, None, out, None, ws, 0)
    assert len(seen) == 1
