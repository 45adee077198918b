"""Pyramid and Scharr tiles at the image's edges: widths around the 16-byte
chunk, the tile and its halo, from 1 px up, through the single build, the
batched launches built in place (aligned rows of any width) and from a caller
image.  Integer arithmetic, compared for equality."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

WIDTHS = [1, 2, 3, 4, 5, 15, 16, 17, 63, 65, 127, 128, 129, 130, 131, 143, 145, 160, 161, 257]


@pytest.mark.parametrize("h", [1, 2, 5, 31, 34, 67, 131])
@pytest.mark.parametrize("grad", [1, 2, 0])
def test_every_width(h, grad):
    import torch

    import paper_2607_01757_gb300 as vt

    rng = np.random.Generator(np.random.PCG64(h * 3 + grad))
    imgs = [rng.integers(0, 256, (h, w), dtype=np.uint8) for w in WIDTHS]
    levels = [1 + (i % 4) for i in range(len(imgs))]
    dev = [torch.from_numpy(i).cuda() for i in imgs]
    one, place, copy = ([vt.vt_pyramid_create(i.shape[1], h, L) for i, L in zip(imgs, levels)] for _ in range(3))
    for d, L, p in zip(dev, levels, one):
        if grad:
            vt.vt_pyramid_build_grad(d, L, grad, out=p)
        else:
            vt.vt_pyramid_build(d, L, out=p)
    for d, p in zip(dev, place):
        vt.vt_pyramid_upload(p, d)
    b = vt.Batch(2 * len(imgs), 1)
    jobs = [vt.frame_job(p.level(0), p) for p in place] + [vt.frame_job(d, p) for d, p in zip(dev, copy)]
    vt.vt_batch_set(b, jobs, [], vt.KltParams(levels=1), grad_type=grad)
    vt.vt_batch_run(b)
    torch.cuda.synchronize()
    for img, L, trio in zip(imgs, levels, zip(one, place, copy)):
        ref = oracle.build_pyramid(img, L)
        for p in trio:
            for l in range(L):
                assert np.array_equal(p.level(l).cpu().numpy(), ref.levels[l]), (img.shape, l)
                if grad == 1:
                    g = p.grad(l).cpu().numpy()
                    assert np.array_equal(g[..., 0], ref.gx[l]) and np.array_equal(g[..., 1], ref.gy[l]), (img.shape, l)
                elif grad == 2:
                    g = p.grad(l).cpu().numpy()
                    ex = np.stack([ref.gx[l], ref.gy[l]], -1).astype(np.float32) / 32
                    assert np.array_equal(g.view(np.uint16), ex.astype(np.float16).view(np.uint16)), (img.shape, l)
    b.free()


@pytest.mark.parametrize("grad", [1, 0])
def test_pinned_host_images(grad):
    """Pinned host frames, read by the first launch (small ones, and rows that
    need a new pitch) or copied up (a large frame in one piece), rewritten on
    the host between builds; and a pageable one."""
    import torch

    import paper_2607_01757_gb300 as vt

    rng = np.random.Generator(np.random.PCG64(grad))
    for w, h, L in [(1, 1, 1), (63, 40, 2), (128, 96, 1), (641, 479, 4), (704, 300, 3), (1280, 1024, 3), (1283, 900, 2)]:
        pin = torch.empty((h, w), dtype=torch.uint8, pin_memory=True)
        p = vt.vt_pyramid_create(w, h, L)
        for k in range(3):
            img = rng.integers(0, 256, (h, w), dtype=np.uint8)
            src = pin if k < 2 else torch.from_numpy(img)
            src.copy_(torch.from_numpy(img))
            if grad:
                vt.vt_pyramid_build_grad(src, L, vt.VT_GRAD_S16, out=p)
            else:
                vt.vt_pyramid_build(src, L, out=p)
            torch.cuda.synchronize()
            ref = oracle.build_pyramid(img, L)
            for l in range(L):
                assert np.array_equal(p.level(l).cpu().numpy(), ref.levels[l]), (w, h, k, l)
                if grad:
                    g = p.grad(l).cpu().numpy()
                    assert np.array_equal(g[..., 0], ref.gx[l]) and np.array_equal(g[..., 1], ref.gy[l]), (w, h, k, l)
