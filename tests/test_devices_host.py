"""Every call works on each device of a process: what a kernel is allowed on one
device (dynamic shared memory above 48 KB) is asked for on the next as well."""

import ctypes as C

import numpy as np

import paper_2607_01757_gb300.vt as vt
from fake_lib import load


def test_calls_on_two_devices():
    lib = load()
    for f in ("vt_gftt_free", "vt_batch_free", "vt_pyramid_free"):
        getattr(lib, f).restype = None
    img = np.zeros((480, 752), np.uint8)
    pts = np.zeros((8, 2), np.float32)
    st = np.zeros(8, np.uint8)
    cnt = np.zeros(4, np.int32)
    p = lambda a: C.c_void_p(a.ctypes.data)  # noqa: E731

    for dev in (0, 1, 0, 5):
        lib.fake_set_device(dev)
        pyr = [C.c_void_p() for _ in range(3)]
        assert lib.vt_pyramid_build(p(img), 752, 480, 752, 4, 1, None, C.byref(pyr[2])) == 0
        for t in (1, 2, 1):
            for h in pyr[:2]:
                assert lib.vt_pyramid_build_grad(p(img), 752, 480, 752, 4, 1, t, None, C.byref(h)) == 0, (dev, t)
        for win in (9, 15, 21, 31):
            for min_eig in (1e-4, 1e-6):
                prm = vt.KltParams(win=win, min_eig=min_eig).c()
                assert lib.vt_klt_track_ex(pyr[0], pyr[1], p(pts), 8, None, C.byref(prm), p(pts), p(st), None, None,
                                           None) == 0, (dev, win)
                assert lib.vt_klt_track_fb(pyr[0], pyr[1], p(pts), 8, C.byref(prm), p(pts), p(st), None, None,
                                           None) == 0, (dev, win)
                b = C.c_void_p()
                assert lib.vt_batch_create(2, 2, C.byref(b)) == 0
                fr = vt.vt_frame_job(img.ctypes.data, 752, pyr[1].value)
                tk = vt.vt_track_task(pyr[0].value, pyr[1].value, pts.ctypes.data, 8, 1, pts.ctypes.data, st.ctypes.data,
                                      None, None, None, 0, None)
                for warps in (4, 8):
                    assert lib.vt_batch_config(b, warps, 0, 0) == 0
                    assert lib.vt_batch_set(b, C.byref(fr), 1, 1, C.byref(tk), 1, C.byref(prm)) == 0
                    assert lib.vt_batch_run(b, None) == 0, (dev, win, warps)
                assert lib.vt_klt_track_tasks_noalloc(C.byref(tk), 1, C.byref(prm), None) == 0
                lib.vt_batch_free(b)
        g = C.c_void_p()
        assert lib.vt_gftt_create(752, 480, C.byref(g)) == 0
        gp = vt.GfttParams(max_corners=8).c()
        assert lib.vt_gftt_detect(g, pyr[0], 0, C.byref(gp), None, 0, p(pts), None, p(cnt), None) == 0, dev
        lib.vt_gftt_free(g)
        ids = np.zeros(8, np.int32)
        pool = vt.vt_track_pool(pts.ctypes.data, ids.ctypes.data, ids.ctypes.data, cnt.ctypes.data, cnt[1:].ctypes.data, 8)
        job = vt.vt_carry_job(pool, pts.ctypes.data, st.ctypes.data, None)
        assert lib.vt_tracks_carry(C.byref(job), 1, C.c_float(10.0), None) == 0, dev
        for h in pyr:
            lib.vt_pyramid_free(h)
        assert lib.fake_refused() == 0, dev
    assert lib.fake_launches() > 200
