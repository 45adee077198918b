"""Two shortcuts of the tracker.  The eigenvalue test is decided from a bound
unless the caller reads lambda_min: with and without it, everything else is the
same bit for bit, around thresholds that many points fail.  The moments of
footprint cells that a position left are kept: with eps 0 every point takes all
30 iterations, many of them hovering at a cell's edge, and still agrees with
the oracle."""

import numpy as np
import pytest

import oracle
import synth
from parity import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cfg():
    return synth.make_config1(7, n=400)


def _track(vt, torch, I, J, pts, prm, **kw):
    n = len(pts)
    o = dict(out=torch.zeros((n, 2), device="cuda"), st=torch.zeros(n, dtype=torch.uint8, device="cuda"),
             err=torch.zeros(n, device="cuda"), rs=torch.zeros(n, dtype=torch.uint8, device="cuda"),
             it=torch.zeros(n, dtype=torch.int32, device="cuda"))
    vt.vt_klt_track_ex(I, J, pts, prm, o["out"], o["st"], o["err"], reason=o["rs"], iters=o["it"], **kw)
    return o


@pytest.mark.parametrize("win", [9, 15, 21, 31])
@pytest.mark.parametrize("grad", [0, 1, 2])
def test_lambda_min_wanted_or_not(cfg, win, grad):
    import torch

    import paper_2607_01757_gb300 as vt

    I, J = (vt.vt_pyramid_build_grad(i, 4, grad) if grad else vt.vt_pyramid_build(i, 4) for i in (cfg.I, cfg.J))
    pts = torch.from_numpy(cfg.pts).cuda()
    lm = torch.zeros(len(pts), device="cuda")
    _track(vt, torch, I, J, pts, vt.KltParams(win=win, levels=4), lmin=lm)
    lost = 0
    for q in (0.05, 0.5, 0.9):
        thr = max(6e-5, float(torch.quantile(lm, q)))  # (from 5e-5 on no level needs FP64)
        prm = vt.KltParams(win=win, levels=4, min_eig=thr)
        a = _track(vt, torch, I, J, pts, prm)
        b = _track(vt, torch, I, J, pts, prm, lmin=torch.zeros(len(pts), device="cuda"))
        for k in a:
            assert torch.equal(a[k], b[k]), (q, k)
        lost += int((a["rs"] == vt.VT_LOST_EIG).sum())
    assert lost > 100


@pytest.mark.parametrize("win,levels", [(9, 3), (21, 4)])
def test_every_iteration_taken(cfg, win, levels):
    import torch

    import paper_2607_01757_gb300 as vt

    I, J = (vt.vt_pyramid_build_grad(i, levels, vt.VT_GRAD_S16) for i in (cfg.I, cfg.J))
    o = _track(vt, torch, I, J, torch.from_numpy(cfg.pts).cuda(), vt.KltParams(win=win, levels=levels, eps=0.0))
    r = oracle.track(oracle.build_pyramid(cfg.I, levels), oracle.build_pyramid(cfg.J, levels), cfg.pts, win, levels,
                     30, 0.0, 1e-4)
    compare(o["out"].cpu().numpy(), o["st"].cpu().numpy(), o["rs"].cpu().numpy(), r, "eps 0")
    assert np.array_equal(np.unique(o["it"].cpu().numpy()[o["st"].cpu().numpy() == 1]), [30 * levels])
