"""A batched step repeated gives the same bits every time, and the bits of the
single calls on the same images: positions, statuses and errors.  On a
difference the message names the point, and says whether the pyramids under it
were the same."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(640, 480), (752, 480), (961, 600), (1439, 1077), (1920, 1200), (200, 150), (97, 65), (1283, 1000)]


def _images(w, h, seed, torch):
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    t = torch.zeros((1, 1, h + 32, w + 32), device="cuda")
    for s in (2, 4, 8, 16):
        n = torch.randn((1, 1, (h + 32) // s + 2, (w + 32) // s + 2), generator=g, device="cuda")
        t += s**0.5 * 9.0 * torch.nn.functional.interpolate(n, size=(h + 32, w + 32), mode="bicubic", align_corners=False)
    t = t[0, 0] + 128.0
    a, b = t[16:16 + h, 16:16 + w], t[14:14 + h, 19:19 + w]
    return [(x + torch.randn((h, w), generator=g, device="cuda")).round().clamp(0, 255).to(torch.uint8).contiguous()
            for x in (a, b)], g


def test_repeated_steps_and_single_calls():
    import torch

    import paper_2607_01757_gb300 as vt

    prm = vt.KltParams(win=21, levels=4)
    streams, frames, tasks = [], [], []
    for k in range(32):
        w, h = SHAPES[k % len(SHAPES)]
        img, g = _images(w, h, k, torch)
        n = 200 + 57 * k
        pts = torch.rand((n, 2), generator=g, device="cuda") * torch.tensor([w - 1.0, h - 1.0], device="cuda")
        L = 4 + k % 3
        pyr = [vt.vt_pyramid_create(w, h, L) for _ in range(2)]
        out = [torch.zeros((n, 2), device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda"), torch.zeros(n, device="cuda")]
        streams.append((img, pts, pyr, out, L))
        frames += [vt.frame_job(i, p) for i, p in zip(img, pyr)]
        tasks.append(vt.track_task(pyr[0], pyr[1], pts, *out, fb=True, levels=L))
    want = []
    for img, pts, _, out, L in streams:
        one = [vt.vt_pyramid_build_grad(i, L, vt.VT_GRAD_S16) for i in img]
        ref = [torch.zeros_like(o) for o in out]
        vt.vt_klt_track_fb(one[0], one[1], pts, vt.KltParams(win=21, levels=L), *ref)
        want.append((one, ref))
    tracked = sum(int(r[1].sum()) for _, r in want)
    total = sum(len(s[1]) for s in streams)
    assert tracked > 0.5 * total, (tracked, total)
    b = vt.Batch(len(frames), len(tasks))
    for rep in range(100):
        for _, _, _, out, _ in streams:
            for o in out:
                o.zero_()
        vt.vt_batch_set(b, frames, tasks, prm)
        (vt.vt_batch_run_graph if rep % 2 else vt.vt_batch_run)(b)
        for k, ((img, pts, pyr, out, L), (one, ref)) in enumerate(zip(streams, want)):
            for name, o, r in zip(("position", "status", "error"), out, ref):
                if not torch.equal(o, r):
                    i = int(torch.nonzero((o != r).reshape(len(pts), -1).any(1))[0])
                    same = all(torch.equal(p.level(l), q.level(l)) and torch.equal(p.grad(l), q.grad(l))
                               for p, q in zip(pyr, one) for l in range(L))
                    pytest.fail(f"step {rep}, stream {k}: {name} of point {i} at {pts[i].tolist()}: {o[i].tolist()}, single "
                                f"call {r[i].tolist()}; level-0 results {out[0][i].tolist()} {ref[0][i].tolist()}; pyramids "
                                f"{'the same' if same else 'differ'}")
    b.free()
