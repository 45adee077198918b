"""The gate at the ends of its parameters: infinite thresholds, rigs in other
units, rotations scaled out of FP32's range, far points.  Decisions equal the
oracle's outside its margin; what the earlier all-FP64 route settled in one pass
is not settled in two."""

import numpy as np
import pytest

from oracle import stereo as S
from test_gpu_stereo_gate import MARGIN, _gpu_gate, _rot

pytestmark = pytest.mark.gpu


def _pairs(n, baseline, seed, depth=600.0, noise=0.4, scale=1.0):
    """Pairs of a rig whose translation is `baseline` long; the scene in baselines
    is the same for every length.  scale: R and t together."""
    rng = np.random.Generator(np.random.PCG64(seed))
    d = np.array([-1.0, 0.05, -0.02]) / np.linalg.norm([-1.0, 0.05, -0.02])
    rig = S.Rig(kl=(458.7, 457.3, 367.2, 248.4), kr=(520.0, 519.0, 379.9, 255.2), R=_rot(0.01, -0.02, 0.005),
                t=baseline * d)
    z = np.exp(rng.uniform(np.log(2.0), np.log(depth), n))
    XL = np.stack([rng.uniform(-0.5, 0.5, n) * z, rng.uniform(-0.4, 0.4, n) * z, z], 1)
    XR = XL @ rig.R.T + d
    pl = np.stack([rig.kl[0] * XL[:, 0] / z + rig.kl[2], rig.kl[1] * XL[:, 1] / z + rig.kl[3]], 1)
    pr = np.stack([rig.kr[0] * XR[:, 0] / XR[:, 2] + rig.kr[2], rig.kr[1] * XR[:, 1] / XR[:, 2] + rig.kr[3]], 1)
    pr += rng.normal(0, noise, pr.shape)
    rig.R, rig.t = rig.R * scale, rig.t * scale
    return pl.astype(np.float32), pr.astype(np.float32), rig


def _same(pl, pr, rig, prm):
    r = S.stereo_gate(pl, pr, None, rig, prm)
    xyz, st, rs = _gpu_gate(pl, pr, None, rig, prm)
    bad = (rs != r.reason) & ~(r.margin < MARGIN)
    assert not bad.any(), (np.nonzero(bad)[0][:8], rs[bad][:8], r.reason[bad][:8], r.margin[bad][:8])
    assert (st == (rs == S.GATE_OK)).all()
    return r, xyz, rs


def _us(pl, pr, rig, prm):
    import torch

    import paper_2607_01757_gb300 as vt

    n = len(pl)
    a, b = torch.from_numpy(pl).cuda(), torch.from_numpy(pr).cuda()
    st = torch.zeros(n, dtype=torch.uint8, device="cuda")
    R = vt.StereoRig(rig.kl, rig.kr, rig.R, rig.t)
    P = vt.GateParams(prm.min_disp, prm.z_min, prm.z_max, prm.max_reproj)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(7):
        e0.record()
        for _ in range(5):
            vt.vt_stereo_gate(a, b, R, P, st)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 200)
    return best


@pytest.mark.parametrize("min_disp", [0.0, 1.0, 1e200, np.inf])
@pytest.mark.parametrize("max_reproj", [0.0, 1.5, 1e200, np.inf])
def test_infinite_thresholds(min_disp, max_reproj):
    pl, pr, rig = _pairs(3000, 0.11, 1)
    r, _, rs = _same(pl, pr, rig, S.GateParams(min_disp, 0.3, np.inf, max_reproj))
    if min_disp > 1e100:
        assert (rs == S.GATE_DISP).all()
    elif max_reproj > 1e100:
        assert not (rs == S.GATE_REPROJ).any() and (rs == S.GATE_OK).sum() > 1000


def test_infinite_thresholds_time():
    """A bound that nothing reaches leaves no pair to the slow route (which takes
    six times as long for all of them)."""
    pl, pr, rig = _pairs(200000, 0.11, 2)
    with_bound = _us(pl, pr, rig, S.GateParams(1.0, 0.3, np.inf, 3.0))
    without = _us(pl, pr, rig, S.GateParams(1.0, 0.3, np.inf, np.inf))
    assert without < 2.0 * with_bound, (without, with_bound)


@pytest.mark.parametrize("scale", [1e-39, 1e-20, 1e6, 1e20, 1e39])
def test_rotation_out_of_range(scale):
    """R and t scaled together describe the same rig up to the scale of X_R: the
    disparity is the unscaled one's (FP32 reciprocals and rotation angles must not
    decide it)."""
    pl, pr, rig = _pairs(2000, 0.11, 3, scale=scale)
    pr[:50] = np.float32([rig.kr[2], rig.kr[3]])  # (the principal point: 0 / 0 where a ray's depth is lost)
    prm = S.GateParams(20.0, 0.3, 50.0, 1.5)
    r = S.stereo_gate(pl, pr, None, rig, prm)
    _, _, rs = _gpu_gate(pl, pr, None, rig, prm)
    far = np.abs(r.disparity - prm.min_disp) > MARGIN
    assert (50 < (r.reason == S.GATE_DISP).sum() < 1950)
    assert ((rs == S.GATE_DISP) == (r.reason == S.GATE_DISP))[far].all()
