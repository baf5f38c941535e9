"""The numpy views that results are handed out as: in place, writable, of the
right length and type; copies and empty columns on their own."""
import numpy as np
import pytest

from paper_2004_04334_gb300 import hp


@pytest.mark.parametrize("dtype", [np.uint16, np.int32, np.uint32, np.float32, np.uint64])
@pytest.mark.parametrize("n", [1, 7, 4096])
def test_view_and_copy(dtype, n):
    base = np.arange(n + 1).astype(dtype)
    view = hp._arr(base.ctypes.data, n, dtype, copy=False)
    copy = hp._arr(base.ctypes.data, n, dtype)
    assert view.dtype == dtype and view.shape == (n,) and view.flags.writeable and copy.flags.writeable
    assert np.array_equal(view, base[:n]) and np.array_equal(copy, base[:n])
    view[n - 1] = 9
    assert base[n - 1] == 9 and base[n] == n and copy[n - 1] == dtype(n - 1)


def test_empty():
    for ptr, n in ((None, 0), (None, 5), (4096, 0)):
        a = hp._arr(ptr, n, np.int32)
        assert a.dtype == np.int32 and a.shape == (0,)
