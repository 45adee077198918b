"""Detector calls whose candidates crowd: no or little local suppression, so that
nearly every pixel is one (lists longer than what the selection works on at a
time), distances that span many or few of the grid's cells, ties.  The same
corners as the greedy in priority order, and a time of its order."""

import numpy as np
import pytest

from test_gpu_gftt_strips import _same

pytestmark = pytest.mark.gpu


def _noise(w, h, seed):
    return np.random.Generator(np.random.PCG64(seed)).integers(0, 256, (h, w), dtype=np.uint8)


def _dots(w, h):
    yy, xx = np.mgrid[0:h, 0:w]
    return np.where((xx % 6 == 2) & (yy % 6 == 3), 200, 20).astype(np.uint8)


@pytest.mark.parametrize("min_dist", [1, 2, 3, 10, 30, 100])
@pytest.mark.parametrize("nms", [0, 1])
@pytest.mark.parametrize("corners", [64, 8192])
def test_dense_candidates(min_dist, nms, corners):
    import paper_2607_01757_gb300 as vt

    prm = vt.GfttParams(max_corners=corners, quality=0.0, min_dist=min_dist, nms_radius=nms, block_radius=1, border=1)
    _same([_noise(64, 48, 1), _dots(64, 48), _noise(181, 67, 2)], prm)


@pytest.mark.parametrize("min_dist,corners", [(1, 8192), (2, 8192), (5, 8192), (40, 8192), (3, 500)])
def test_long_lists(min_dist, corners):
    """More local maxima than are worked on at a time, with distinct scores and
    with a handful of them."""
    import paper_2607_01757_gb300 as vt

    prm = vt.GfttParams(max_corners=corners, quality=0.0, min_dist=min_dist, nms_radius=0, block_radius=1, border=0)
    few = (_noise(300, 240, 5) // 64 * 80).astype(np.uint8)
    _same([_noise(300, 240, 4), few], prm)


def test_time():
    """Without local suppression, 8,192 corners of a 752 x 480 frame take a few
    milliseconds at most, as they did when the whole grid selected them."""
    import torch

    import paper_2607_01757_gb300 as vt

    pyr = vt.vt_pyramid_build_grad(_noise(752, 480, 3), 1, vt.VT_GRAD_S16)
    g = vt.Gftt(752, 480)
    xy, cnt = torch.zeros((8192, 2), device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for md, limit in ((1, 2.0), (30, 2.5)):
        best = float("inf")
        for _ in range(5):
            a.record()
            vt.vt_gftt_detect(g, pyr, 0, vt.GfttParams(max_corners=8192, quality=0.0, min_dist=md, nms_radius=0), xy, cnt)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        assert best < limit, (md, best)
    g.free()
