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


def _points(pl, pr, rig):
    """The triangulated points to better than 1e-9 of their distance whatever the
    rig's unit: inverse iteration on the generalised problem, the last coordinate
    scaled to the translation, from the FP64 SVD's vector."""
    L, Q = pl.astype(np.float64), pr.astype(np.float64)
    xl = (L - rig.kl[2:]) / rig.kl[:2]
    xr = (Q - rig.kr[2:]) / rig.kr[:2]
    x = S.triangulate_dlt(xl, xr, rig.R, rig.t)
    unit = np.linalg.norm(rig.t)
    o, z = np.ones(len(pl)), np.zeros(len(pl))
    P = np.concatenate([rig.R, rig.t[:, None] / unit], 1)
    A = np.stack([np.stack([-o, z, xl[:, 0], z], 1), np.stack([z, -o, xl[:, 1], z], 1), xr[:, :1] * P[2] - P[0],
                  xr[:, 1:] * P[2] - P[1]], 1)
    B = np.array([1.0, 1.0, 1.0, unit**-2])
    y = x * np.array([1.0, 1.0, 1.0, unit])
    M = np.einsum("nri,nrj->nij", A, A)
    for _ in range(3):
        lam = ((A @ y[..., None])[..., 0]**2).sum(1) / (B * y * y).sum(1)
        K = M - 0.999 * lam[:, None, None] * np.diag(B)
        y = np.linalg.solve(K, (B * y)[..., None])[..., 0]
        y /= np.linalg.norm(y, axis=1)[:, None]
    return unit * y[:, :3] / y[:, 3:]


BASELINES = [1e-3, 0.015, 0.016, 0.11, 1.9, 2.0, 11.0, 110.0, 250.0, 1000.0, 3e4]


@pytest.mark.parametrize("baseline", BASELINES)
@pytest.mark.parametrize("depth", [600.0, 5e4])
def test_units(baseline, depth):
    """The same scene in any unit of length, near and far.  The fast route's points
    are off by at most its guard, 3e-8 of their distance, besides the output's
    rounding; a pair in a thousand may be left to the other route (whose error
    grows with the translation)."""
    n = 5000
    pl, pr, rig = _pairs(n, baseline, int(depth), depth=depth, noise=0.4 if depth < 1e3 else 0.002)
    r, xyz, rs = _same(pl, pr, rig, S.GateParams(0.0, 0.0, np.inf, 1.5))
    if baseline < 0.0157:  # the FP64 route alone
        return
    X = _points(pl, pr, rig)
    tri = (rs == S.GATE_OK) | (rs == S.GATE_DEPTH) | (rs == S.GATE_REPROJ)
    tri &= (np.abs(X) < 1e5 * baseline).all(1)  # (noise puts far points anywhere; beyond the guard there is the other route)
    tol = 2.0**-24 * np.abs(X) + 3e-8 * (2.0 * baseline + np.abs(X).sum(1))[:, None]
    off = (np.abs(xyz - X) > tol).any(1) & tri
    assert tri.sum() > 0.5 * n and off.sum() <= 0.001 * n, (off.sum(), (np.abs(xyz - X) / tol)[tri].max())


def test_units_time():
    """... and in the same time."""
    us = {b: _us(*_pairs(200000, b, 5), S.GateParams(1.0, 0.1 * b, 500.0 * b, 1.5)) for b in (0.11, 110.0, 500.0, 3e4)}
    assert all(v < 1.5 * us[0.11] for v in us.values()), us
