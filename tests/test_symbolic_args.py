"""Row pointers that do not ascend are refused by the device symbolic phase
before anything is read through them: the last one may address far more columns
than the caller's array holds.  No CUDA call is made on this path."""
from __future__ import annotations

import ctypes as C

import numpy as np
import pytest


@pytest.mark.parametrize("rp", [[0, 2, 1, 3], [0, 3, 2, 1 << 30], [0, 1, -1, 4], [0, 1, 5, 3]])
def test_descending_row_pointers(libbilu, rp):
    from paper_1703_01325_gb300 import _lib as L
    out = C.c_void_p()
    keep = [np.array(rp, np.int32), np.array([0, 1, 2], np.int32)]
    p = [a.ctypes.data_as(C.POINTER(C.c_int32)) for a in keep]
    for call in (lambda: libbilu.bilu_symbolic(3, *p, 1, C.byref(out)),
                 lambda: libbilu.bilu_symbolic_gpu(3, *p, 1, 64, None, C.byref(out))):
        assert call() == L.BILU_ERR_PATTERN
        assert not out.value
