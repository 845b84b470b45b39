"""What the binding takes as a host int32 list, and what it refuses (no GPU needed: the library
is called without a context and answers that, once the arguments are through)."""
import ctypes

import numpy as np
import pytest

from paper_2609_31224_gb300 import _lib as L
from paper_2609_31224_gb300 import build as B


@pytest.fixture(scope="module")
def lib():
    B.build()
    return L.load_library()


@pytest.mark.parametrize("a,want", [
    (3, [3]), (np.int32(3), [3]), (np.array(3, np.int32), [3]), ([1, 2], [1, 2]),
    (range(3), [0, 1, 2]), (np.arange(4, dtype=np.int64), [0, 1, 2, 3]),
    (np.arange(6, dtype=np.int32)[::2], [0, 2, 4]), (np.arange(3, dtype=">i4"), [0, 1, 2]),
])
def test_int32_lists(a, want):
    got, ptr = L.host_i32(a)
    assert got.ndim == 1 and got.dtype == np.int32 and got.flags.c_contiguous
    assert len(got) == len(want) and [ptr[i] for i in range(len(want))] == want


def test_an_int32_array_is_passed_as_it_is():
    a = np.arange(4, dtype=np.int32)
    assert L._i32(a) is a


def _calls(lib, p):
    return [lambda: lib.kvc_append_chunk(None, 1, p, p, None, None, None, None),
            lambda: lib.kvc_evict(None, 1, p, None, None), lambda: lib.kvc_release(None, 1, p, None)]


def test_typed_pointers_are_checked(lib):
    """The raw calls take int32 pointers and refuse what is not one."""
    ok = [L.host_i32([0, 1])[1], (ctypes.c_int32 * 2)(0, 1), None]
    wrong = [np.zeros(2, np.int64).ctypes.data_as(ctypes.POINTER(ctypes.c_int64)),
             (ctypes.c_int64 * 2)(0, 1), (ctypes.c_float * 2)(), b"01234567", 4096]
    for p in ok:
        for call in _calls(lib, p):
            assert call() != 0  # KVC_EINVAL: no context
    for p in wrong:
        for call in _calls(lib, p):
            with pytest.raises(ctypes.ArgumentError):
                call()
