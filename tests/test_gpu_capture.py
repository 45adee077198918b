"""The single-pair calls captured into a user's CUDA graph: a build from a
device image, forward-backward tracking and detection, replayed on new input,
equal the same calls issued directly."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_build_track_detect_in_a_user_graph():
    import torch

    import paper_2607_01757_gb300 as vt

    a, b = synth.make_config1(1), synth.make_config1(2)
    L, n = 4, 150
    prm = vt.KltParams(win=21, levels=L)
    img = [torch.from_numpy(x).cuda() for x in (a.I, a.J)]
    pts = torch.from_numpy(a.pts).cuda()
    g = vt.Gftt(752, 480)

    def bufs():
        return dict(pyr=[vt.vt_pyramid_create(752, 480, L) for _ in range(2)], out=torch.zeros((n, 2), device="cuda"),
                    st=torch.zeros(n, dtype=torch.uint8, device="cuda"), err=torch.zeros(n, device="cuda"),
                    xy=torch.zeros((n, 2), device="cuda"), cnt=torch.zeros(1, dtype=torch.int32, device="cuda"))

    def work(d):
        for i, p in zip(img, d["pyr"]):
            vt.vt_pyramid_build_grad(i, L, vt.VT_GRAD_S16, out=p)
        vt.vt_klt_track_fb(d["pyr"][0], d["pyr"][1], pts, prm, d["out"], d["st"], d["err"])
        vt.vt_gftt_detect(g, d["pyr"][1], 0, vt.GfttParams(max_corners=n), d["xy"], d["cnt"], mask=d["out"])

    ref, cap = bufs(), bufs()
    work(ref)  # (and the first call's one-time setup)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        work(cap)
    for frames in (a, b):
        img[0].copy_(torch.from_numpy(frames.I))
        img[1].copy_(torch.from_numpy(frames.J))
        pts.copy_(torch.from_numpy(frames.pts))
        work(ref)
        torch.cuda.synchronize()
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        for k in ("out", "st", "err", "xy", "cnt"):
            assert torch.equal(ref[k], cap[k]), k
        for l in range(L):
            assert torch.equal(ref["pyr"][1].level(l), cap["pyr"][1].level(l))
            assert torch.equal(ref["pyr"][1].grad(l), cap["pyr"][1].grad(l))
    assert int(ref["st"].sum()) > 100 and int(ref["cnt"].item()) == np.minimum(n, int(ref["cnt"].item()))
