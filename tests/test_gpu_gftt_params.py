"""The ends of the detector's parameters -- minimum distances whose square passes
32 bits, levels wide enough for squared distances that do, qualities from zero
to infinity --: masks and selection, compared for equality."""

import numpy as np
import pytest

from test_gpu_gftt_strips import _same

pytestmark = pytest.mark.gpu


def _frame(w, h, seed):
    return np.random.Generator(np.random.PCG64(seed)).integers(0, 256, (h, w), dtype=np.uint8)


@pytest.mark.parametrize("min_dist", [46340, 46341, 65536, 131072, 1 << 20, 2**31 - 1])
@pytest.mark.parametrize("nms", [4, 6])
def test_mask_points(min_dist, nms):
    """A mask point inside the level masks all of it; one about min_dist away
    masks the part on its side; non-finite ones mask nothing."""
    import paper_2607_01757_gb300 as vt

    prm = vt.GfttParams(max_corners=50, quality=0.0, min_dist=min_dist, nms_radius=nms, border=2)
    f = np.float32
    masks = [np.array([[20.0, 30.0]], f), np.array([[160.5 - min_dist, 48.0]], f),
             np.array([[160.0, 48.5 + min_dist], [np.nan, 3.0]], f), np.array([[np.inf, 3.0], [5.0, -np.inf]], f),
             np.array([[3.0 * min_dist, -3.0 * min_dist]], f)]
    imgs = [_frame(320, 96, min_dist % 97 + k) for k in range(len(masks))]
    _same(imgs, prm, masks)


@pytest.mark.parametrize("min_dist", [200, 23171, 30000, 46341, 50000, 65534])
def test_wide_level(min_dist):
    import paper_2607_01757_gb300 as vt

    prm = vt.GfttParams(max_corners=40, quality=0.3, min_dist=min_dist, nms_radius=4, border=1)
    _same([_frame(65535, 12, 3)], prm)
    _same([_frame(12, 65535, 4)], prm, [np.array([[6.0, 2000.0]], np.float32)])


@pytest.mark.parametrize("quality", [0.0, -0.0, 1e-45, 1.0, 1.5, float("inf")])
@pytest.mark.parametrize("nms", [2, 4])
def test_quality_at_its_ends(quality, nms):
    """Both zeros admit every local maximum, 1 the frame's best, more none."""
    import paper_2607_01757_gb300 as vt

    prm = vt.GfttParams(max_corners=300, quality=quality, min_dist=5, nms_radius=nms)
    _same([_frame(320, 200, 1), np.full((60, 80), 9, np.uint8)], prm)
