"""vktStructuredVolumeCreateViews / vktStructuredVolumesDestroy: argument checks, all or none.
Needs no device."""
import ctypes
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2203_10213_gb300._lib import load  # noqa: E402


@pytest.mark.parametrize("bad", [(0, 4, 4), (4, -1, 4)])
def test_all_or_none(bad):
    lib = load()
    out = (ctypes.c_void_p * 2)(1, 1)
    ptrs = (ctypes.c_void_p * 2)(None, None)
    dims = (ctypes.c_int32 * 6)(4, 4, 4, *bad)
    args = (dims, 2, 1.0, 1.0, 1.0, 0.0, 1.0)
    assert lib.vktStructuredVolumeCreateViews(0, out, ptrs, *args) == 1
    assert lib.vktStructuredVolumeCreateViews(2, None, ptrs, *args) == 1
    assert lib.vktStructuredVolumeCreateViews(2, out, ptrs, *args) == 1     # NULL pointers, bad dims
    assert not out[0] and not out[1]
    assert lib.vktStructuredVolumesDestroy(0, out) == 1
    assert lib.vktStructuredVolumesDestroy(2, None) == 1
    assert lib.vktStructuredVolumesDestroy(2, out) == 2                     # NULL handles
