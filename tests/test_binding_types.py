"""The binding refuses arrays of another type than the entry point takes (no GPU)."""
import ctypes

import numpy as np
import pytest

from paper_1412_1127_gb300 import _native


@pytest.fixture(scope="module")
def L():
    import __graft_entry__ as g
    g.build()
    return _native.lib()


def clause():
    c = _native.Clause()
    c.op, c.acc_type, c.init, c.out = 0, 0, None, 1
    return c


WRONG = [(ctypes.c_int64 * 8)(), (_native.Region * 1)(), ctypes.pointer(ctypes.c_float(1)), 4096, "clauses", b"", b"x" * 23,
         bytearray(24), [clause()]]


@pytest.mark.parametrize("arg", WRONG, ids=lambda a: type(a).__name__)
def test_clauses_of_another_type_are_refused(L, arg):
    for call in (lambda: L.accr_reduce(None, -1, 0, arg, 1, 0, None),
                 lambda: L.accr_reduce_noalloc(None, -1, 0, arg, 1, 0, None),
                 lambda: L.accr_rowreduce(None, -1, 8, 8, 0, arg, 1, 0, None),
                 lambda: L.accr_segmented_reduce(None, None, -1, 0, arg, 1, 0, None)):
        with pytest.raises(ctypes.ArgumentError):
            call()


def test_clauses_in_every_form_are_taken(L):
    two = (_native.Clause * 2)(clause(), clause())
    for arg in (two, ctypes.byref(two[0]), ctypes.pointer(two[0]), ctypes.cast(two, ctypes.POINTER(_native.Clause)),
                bytes(two), None):
        assert L.accr_reduce(None, -1, 0, arg, 1, 0, None) == _native.ACCR_EINVAL


@pytest.mark.parametrize("arg", [np.arange(4, dtype=np.int32), np.arange(4, dtype=np.uint64), np.arange(4.0),
                                 np.arange(8, dtype=np.int64)[::2], (ctypes.c_int32 * 4)(), 4096, b"x" * 32, [0, 1]],
                         ids=lambda a: str(getattr(a, "dtype", type(a).__name__)))
def test_offsets_of_another_type_are_refused(L, arg):
    with pytest.raises(ctypes.ArgumentError):
        L.accr_segmented_reduce(None, arg, -1, 0, (_native.Clause * 1)(clause()), 1, 0, None)


def test_offsets_in_every_form_are_taken(L):
    cl = (_native.Clause * 1)(clause())
    c = (ctypes.c_int64 * 3)(0, 1, 2)
    for arg in (np.arange(3, dtype=np.int64), c, ctypes.cast(c, ctypes.POINTER(ctypes.c_int64)), None):
        assert L.accr_segmented_reduce(None, arg, -1, 0, cl, 1, 0, None) == _native.ACCR_EINVAL
