"""CPU: result arrays are copied out of the library's memory whole, also where
they pass 2 GiB (the hull vertices of tens of millions of clusters)."""
import ctypes as C

import numpy as np
import pytest

from paper_2510_01592_gb300 import vm


@pytest.mark.parametrize("n", [0, 1, 1000, 2 ** 29 + 3])
def test_copy_of_n_words(n):
    src = np.zeros(max(n, 1), np.int32)
    src[-1] = 7
    ptr = src.ctypes.data_as(C.POINTER(C.c_int32))
    got = vm._copy(ptr, n, vm._I32)
    assert got.shape == (n,) and got.flags.writeable
    if n:
        src[-1] = 8  # the copy is its own
        assert got[-1] == 7 and not got[:min(n - 1, 1000)].any()
