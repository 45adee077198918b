"""How a pinned host frame reaches the device -- read by the first launch where
there is one that needs it, copied where a copy is all the call does -- and how
many launches a build takes: none that has nothing to do."""

import ctypes as C

import numpy as np
import pytest

from fake_lib import load


@pytest.mark.parametrize("w,h,levels,grad,copies,launches", [
    (160, 120, 1, 0, 1, 0), (160, 120, 1, 1, 0, 1), (160, 120, 2, 0, 0, 1), (100, 75, 1, 0, 1, 0), (320, 240, 2, 0, 0, 1),
    (320, 240, 2, 1, 0, 2), (320, 240, 3, 0, 0, 2), (752, 480, 1, 0, 1, 0), (752, 480, 1, 1, 0, 1), (752, 480, 4, 0, 0, 3),
    (752, 480, 4, 1, 0, 3), (1920, 1200, 4, 1, 1, 4), (1919, 1200, 4, 0, 0, 3), (1919, 1200, 4, 1, 0, 4)])
def test_pinned_frame(w, h, levels, grad, copies, launches):
    lib = load()
    lib.vt_pyramid_free.restype = None
    img = np.zeros((h, w), np.uint8)
    lib.fake_pin(C.c_void_p(img.ctypes.data), C.c_size_t(img.nbytes))
    pyr = C.c_void_p()
    before = lib.fake_copies(), lib.fake_launches()
    if grad:
        st = lib.vt_pyramid_build_grad(C.c_void_p(img.ctypes.data), w, h, w, levels, 0, 1, None, C.byref(pyr))
    else:
        st = lib.vt_pyramid_build(C.c_void_p(img.ctypes.data), w, h, w, levels, 0, None, C.byref(pyr))
    assert st == 0 and (lib.fake_copies() - before[0], lib.fake_launches() - before[1]) == (copies, launches)
    if launches == 0:  # built in place: nothing is left to do
        lv = C.c_void_p()
        pitch = C.c_int()
        assert lib.vt_pyramid_level(pyr, 0, C.byref(lv), None, None, C.byref(pitch)) == 0
        assert lib.vt_pyramid_build(lv, w, h, pitch, levels, 1, None, C.byref(pyr)) == 0
        assert (lib.fake_copies() - before[0], lib.fake_launches() - before[1]) == (copies, 0)
    lib.vt_pyramid_free(pyr)
    lib.fake_pin(None, C.c_size_t(0))
