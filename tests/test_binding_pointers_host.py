"""Addresses handed to the ctypes binding are whole numbers (or None for NULL):
objects that ctypes itself would turn into a host address (bytes, str, arrays,
ctypes pointers) are refused before the C call.  The plan handle is NULL here,
so that a call that is made returns EINVAL and touches nothing."""

import ctypes as C
import os

import pytest

import paper_2003_08960_gb300 as ss

pytestmark = pytest.mark.skipif(not os.path.exists(ss._abi.LIB_PATH), reason="libssoct.so is not built")

CALLS = [  # name, number of address arguments, how to call with them
    ("set_workspace", 1, lambda a: ss.ssoct_set_workspace(None, a[0], 0)),
    ("push_frames", 2, lambda a: ss.ssoct_push_frames(None, a[0], 1, True, -1, a[1])),
    ("reconstruct_volume", 3, lambda a: ss.ssoct_reconstruct_volume(None, a[0], a[1], a[2])),
    ("reconstruct_frames", 4, lambda a: ss.ssoct_reconstruct_frames(None, a[0], a[1], a[2], a[3])),
    ("reconstruct_sliding", 3, lambda a: ss.ssoct_reconstruct_sliding(None, a[0], a[1], a[2])),
    ("reconstruct_frames_noalloc", 4, lambda a: ss.ssoct_reconstruct_frames_noalloc(None, a[0], a[1], a[2], a[3])),
    ("get_cuts", 5, lambda a: ss.ssoct_get_cuts(None, a[0], 0, 0, 0, a[1], a[2], a[3], a[4])),
    ("sync", 1, lambda a: ss.ssoct_sync(None, a[0])),
    ("sharpness", 3, lambda a: ss.ssoct_sharpness(None, a[0], a[1], a[2])[0]),
    ("sliding_cuts", 4, lambda a: ss.ssoct_sliding_cuts(None, 0, 0, 0, a[0], a[1], a[2], a[3])),
]


@pytest.mark.parametrize("name,n,call", CALLS, ids=[c[0] for c in CALLS])
def test_addresses_are_whole_numbers(name, n, call):
    good = [4096] * n
    assert call(good) == ss.SSOCT_EINVAL
    assert call([0] * n) == ss.SSOCT_EINVAL and call([None] * n) == ss.SSOCT_EINVAL
    for bad in (b"abc", "abc", 1.5, (C.c_char * 8)(), C.byref(C.c_int()), C.pointer(C.c_int()), C.c_void_p(4096)):
        for k in range(n):
            with pytest.raises((TypeError, C.ArgumentError)):
                call(good[:k] + [bad] + good[k + 1:])
