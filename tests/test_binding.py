"""Array arguments of the Python binding: every form a caller may pass reaches the C call as contiguous values."""
import ctypes as C

import numpy as np
import pytest

from paper_2606_01009_gb300 import melt


def _read_only(a):
    a.setflags(write=False)
    return a


@pytest.mark.parametrize("view,ctype", [(melt._i64, C.c_int64), (melt._i32, C.c_int32)])
@pytest.mark.parametrize("arg", [
    [3, 5, 7],
    (4, 8),
    np.array([1.0, 9.0]),
    np.array([2, 6], dtype=np.int16),
    np.array([2, 6], dtype=">i8"),
    np.arange(12, dtype=np.int64)[::3],
    np.arange(12, dtype=np.int32)[1:7],
    np.arange(6, dtype=np.int64).reshape(2, 3).T,
    _read_only(np.arange(5, dtype=np.int64)),
    _read_only(np.arange(5, dtype=np.int32)),
    np.int64(11),
    [],
])
def test_array_views(view, ctype, arg):
    arr, p = view(arg)
    want = np.atleast_1d(np.asarray(arg)).astype(arr.dtype)
    assert arr.flags.c_contiguous and np.array_equal(arr, want)
    first = C.cast(p if isinstance(p, C._Pointer) else C.byref(p), C.POINTER(ctype))
    flat = want.reshape(-1)
    assert [first[i] for i in range(flat.size)] == flat.tolist()


def test_no_array():
    assert melt._i64(None) == (None, None)
