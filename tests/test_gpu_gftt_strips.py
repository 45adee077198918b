"""Detector strips and chunked selection at their edges: frame sizes around the
strip width and the row groups, every block radius at both strip window radii,
ties (periodic patterns, one crowded score bin) and selections of many chunks.
The result is a list of pixels and FP32 scores, compared for equality."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _same(imgs, prm, masks=None):
    import torch

    import paper_2607_01757_gb300 as vt

    cap = max(1, prm.max_corners)
    g = vt.vt_gftt_create_pixels(sum(i.size for i in imgs))
    pyr = [vt.vt_pyramid_build_grad(np.ascontiguousarray(i), 1, vt.VT_GRAD_S16) for i in imgs]
    xy = torch.zeros((len(imgs), cap, 2), device="cuda")
    sc = torch.zeros((len(imgs), cap), device="cuda")
    cnt = torch.zeros(len(imgs), dtype=torch.int32, device="cuda")
    dm = [None if masks is None or masks[k] is None else torch.from_numpy(masks[k]).cuda() for k in range(len(imgs))]
    jobs = [vt.gftt_job(p, 0, xy[k], cnt[k:k + 1], prm.max_corners, scores_out=sc[k], mask=dm[k])
            for k, p in enumerate(pyr)]
    vt.vt_gftt_detect_many(g, jobs, prm)
    torch.cuda.synchronize()
    for k, img in enumerate(imgs):
        ref = oracle.build_pyramid(np.ascontiguousarray(img), 1)
        rxy, rsc = oracle.gftt(ref.gx[0], ref.gy[0], prm.max_corners, prm.quality, prm.min_dist, prm.nms_radius,
                               prm.block_radius, prm.border,
                               None if dm[k] is None else masks[k].astype(np.float64))
        n = int(cnt[k].item())
        assert n == len(rxy), (img.shape, n, len(rxy))
        assert np.array_equal(xy[k, :n].cpu().numpy(), rxy.astype(np.float32)), img.shape
        assert np.array_equal(sc[k, :n].cpu().numpy().view(np.uint32), rsc.view(np.uint32)), img.shape
    g.free()


@pytest.mark.parametrize("nms", [3, 4])
@pytest.mark.parametrize("br", [0, 1, 2, 3])
def test_strip_edges(nms, br):
    import paper_2607_01757_gb300 as vt

    rng = np.random.Generator(np.random.PCG64(10 * nms + br))
    base = rng.integers(0, 256, (140, 230), dtype=np.uint8)
    flat = (base // 128 * 90).astype(np.uint8)  # few distinct scores: ties inside and across lanes
    shapes = [(1, 1), (2, 9), (7, 3), (8, 112), (9, 113), (63, 111), (64, 224), (65, 225), (67, 119), (140, 230)]
    imgs = [a[:h, :w] for h, w in shapes for a in (base, flat)]
    masks = [rng.uniform(-20, 250, (30, 2)).astype(np.float32) if k % 3 == 0 else None for k in range(len(imgs))]
    prm = vt.GfttParams(max_corners=400, quality=0.0, min_dist=3, nms_radius=nms, block_radius=br, border=1)
    _same(imgs, prm, masks)


@pytest.mark.parametrize("min_dist", [1, 9, 40])
def test_selection_over_many_chunks(min_dist):
    """More candidates than a chunk holds, with distinct scores, with one
    score (a crowded bin that is split by pixel), and strips of every length."""
    import paper_2607_01757_gb300 as vt

    rng = np.random.Generator(np.random.PCG64(min_dist))
    noise = rng.integers(0, 256, (480, 752), dtype=np.uint8)
    yy, xx = np.mgrid[0:480, 0:640]
    dots = np.where((xx % 6 == 2) & (yy % 6 == 3), 200, 20).astype(np.uint8)  # 8,560 equal local maxima
    prm = vt.GfttParams(max_corners=8192, quality=0.0, min_dist=min_dist, nms_radius=4 if min_dist > 1 else 3,
                        block_radius=1, border=2)
    _same([noise, dots], prm)
    _same([synth.make_config1(2).I] * 8 + [noise], vt.GfttParams(max_corners=300, min_dist=min_dist))


@pytest.mark.parametrize("min_dist", [46340, 65536])
def test_min_dist_wider_than_any_level(min_dist):
    """A distance whose square passes 32 bits: the best corner alone is kept,
    also of more candidates than a chunk holds."""
    import paper_2607_01757_gb300 as vt

    rng = np.random.Generator(np.random.PCG64(5))
    prm = vt.GfttParams(max_corners=500, quality=0.0, min_dist=min_dist, nms_radius=3, block_radius=1, border=2)
    _same([rng.integers(0, 256, (480, 752), dtype=np.uint8)], prm)
