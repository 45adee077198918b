"""vt_batch_run_levels_timed takes 4 events and one per pyramid launch, as
vt_batch_info counts them, also of runs that build no pyramid, and records each
of them once."""

import ctypes as C

import numpy as np
import pytest

import paper_2607_01757_gb300.vt as vt
from fake_lib import load


@pytest.mark.parametrize("nframes", [0, 1, 2])
@pytest.mark.parametrize("min_eig", [1e-4, 1e-6])
def test_events(nframes, min_eig):
    lib = load()
    for f in ("vt_batch_free", "vt_pyramid_free"):
        getattr(lib, f).restype = None
    img, pts, st = np.zeros((480, 752), np.uint8), np.zeros((8, 2), np.float32), np.zeros(8, np.uint8)
    pyr = [C.c_void_p() for _ in range(2)]
    for h in pyr:
        assert lib.vt_pyramid_build_grad(C.c_void_p(img.ctypes.data), 752, 480, 752, 4, 1, 1, None, C.byref(h)) == 0
    b, nl = C.c_void_p(), C.c_int()
    assert lib.vt_batch_create(2, 2, C.byref(b)) == 0
    fr = (vt.vt_frame_job * 2)(*[vt.vt_frame_job(img.ctypes.data, 752, h.value) for h in pyr])
    tk = vt.vt_track_task(pyr[0].value, pyr[1].value, pts.ctypes.data, 8, 1, pts.ctypes.data, st.ctypes.data, None, None,
                          None, 0, None)
    prm = vt.KltParams(min_eig=min_eig).c()
    assert lib.vt_batch_set(b, fr, nframes, 1, C.byref(tk), 1, C.byref(prm)) == 0
    assert lib.vt_batch_info(b, None, None, None, C.byref(nl)) == 0
    need = 4 + nl.value - 1 - (min_eig < 5e-5)
    events = (C.c_void_p * 16)(*range(1, 17))
    out = (C.c_void_p * 64)()
    assert lib.vt_batch_run_levels_timed(b, None, events, need - 1) == 1  # VT_ERR_ARG
    for n in (need, need + 1, 16):
        lib.fake_recorded(out)
        assert lib.vt_batch_run_levels_timed(b, None, events, n) == 0, (n, need)
        seen = [out[i] for i in range(lib.fake_recorded(out))]
        want = set(range(1, need + 1)) | ({5} if nframes == 0 and n > 4 else set())
        assert sorted(e for e in seen if e <= 16) == sorted(want)
    lib.vt_batch_free(b)
    for h in pyr:
        lib.vt_pyramid_free(h)
