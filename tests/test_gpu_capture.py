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


def test_captured_detection_finds_the_oracle_corners():
    """What a replayed detection finds is not nothing: the oracle's corners, of
    both frames that pass through the captured image."""
    import torch

    import oracle
    import paper_2607_01757_gb300 as vt

    frames = [synth.make_config1(s).I for s in (1, 2)]
    img = torch.from_numpy(frames[0]).cuda()
    pyr, g, n = vt.vt_pyramid_create(752, 480, 1), vt.Gftt(752, 480), 150
    mask = torch.tensor([[100.0, 100.0], [400.5, 200.25]], device="cuda")
    xy, cnt = torch.zeros((n, 2), device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")

    def work():
        vt.vt_pyramid_build_grad(img, 1, vt.VT_GRAD_S16, out=pyr)
        vt.vt_gftt_detect(g, pyr, 0, vt.GfttParams(max_corners=n), xy, cnt, mask=mask)

    work()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        work()
    for f in (frames[1], frames[0]):
        img.copy_(torch.from_numpy(f))
        xy.zero_()
        cnt.zero_()
        graph.replay()
        torch.cuda.synchronize()
        ref = oracle.build_pyramid(f, 1)
        rxy, _ = oracle.gftt(ref.gx[0], ref.gy[0], n, 0.01, 10, 4, 1, 10, mask.cpu().numpy().astype(np.float64))
        k = int(cnt.item())
        assert k == len(rxy) > 50
        assert np.array_equal(xy[:k].cpu().numpy(), rxy.astype(np.float32))
    g.free()
