"""Builds queued back to back into the same pyramids, each launch starting while
the one before it still runs: what every build leaves is its own image's
pyramid, whatever was there before.  Integer arithmetic, compared for equality."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,levels", [(752, 480, 4), (1920, 1200, 6), (641, 479, 5), (300, 200, 8)])
@pytest.mark.parametrize("grad", [0, 1])
def test_chain(w, h, levels, grad):
    import torch

    import paper_2607_01757_gb300 as vt

    rng = np.random.Generator(np.random.PCG64(w + grad))
    imgs = [rng.integers(0, 256, (h, w), dtype=np.uint8) for _ in range(4)]
    dev = [torch.from_numpy(i).cuda() for i in imgs]
    one = vt.vt_pyramid_create(w, h, levels)
    two = [vt.vt_pyramid_create(w, h, levels) for _ in range(2)]
    b = vt.Batch(2, 1)
    got = []
    for k in range(60):
        i, j = k % 4, (k * 3 + 1) % 4
        if grad:
            vt.vt_pyramid_build_grad(dev[i], levels, vt.VT_GRAD_S16, out=one)
        else:
            vt.vt_pyramid_build(dev[i], levels, out=one)
            vt.vt_gradients(one, vt.VT_GRAD_S16)
        vt.vt_batch_set(b, [vt.frame_job(dev[i], two[0]), vt.frame_job(dev[j], two[1])], [], vt.KltParams(levels=1))
        vt.vt_batch_run(b)
        got.append((i, j, [[(p.level(l).clone(), p.grad(l).clone()) for l in range(levels)] for p in (one, *two)]))
    torch.cuda.synchronize()
    refs = [oracle.build_pyramid(i, levels) for i in imgs]
    want = [[(torch.from_numpy(r.levels[l]).cuda(), torch.from_numpy(np.stack([r.gx[l], r.gy[l]], -1)).cuda())
             for l in range(levels)] for r in refs]
    for k, (i, j, pyr) in enumerate(got):
        for which, p in zip((i, i, j), pyr):
            for l in range(levels):
                assert torch.equal(p[l][0], want[which][l][0]), (k, l)
                assert torch.equal(p[l][1], want[which][l][1]), (k, l)
    b.free()
