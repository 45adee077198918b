"""The gate's two routes (FP32 eigenvectors refined in FP64; all FP64 where that
does not settle a pair) over rigs from a micro-baseline to wide and rotated
ones.  Decisions equal the oracle's outside its margin; a point differs by at
most the float32 rounding of the output (2^-24 relative) plus what FP64
rounding of A^T A does to its null vector: 64 2^-53 |A|^2 / gap for the kernels'
some 60 roundings, plus the 1e-13 at which the refinement stops, carried to the
point through X / X_4."""

import numpy as np
import pytest

from oracle import stereo as S
from test_gpu_stereo_gate import MARGIN, _gpu_gate, _rot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("baseline", [1e-4, 1e-2, 0.11, 2.0, 40.0])
@pytest.mark.parametrize("angle", [0.0, 0.02, 0.5])
@pytest.mark.parametrize("n", [1, 33, 3000])
def test_rigs(baseline, angle, n):
    rng = np.random.Generator(np.random.PCG64(int(1e4 * baseline) + int(100 * angle) + n))
    R = _rot(angle * 0.3, -angle, angle * 0.2)
    d = np.array([-1.0, 0.05, -0.02]) / np.linalg.norm([-1.0, 0.05, -0.02])
    rig = S.Rig(kl=(458.7, 457.3, 367.2, 248.4), kr=(520.0, 519.0, 379.9, 255.2), R=R, t=baseline * d)
    z = baseline * np.exp(rng.uniform(np.log(2.0), np.log(600.0), n))
    XL = np.stack([rng.uniform(-0.5, 0.5, n) * z, rng.uniform(-0.4, 0.4, n) * z, z], 1)
    XR = XL @ R.T + rig.t
    pl = np.stack([rig.kl[0] * XL[:, 0] / z + rig.kl[2], rig.kl[1] * XL[:, 1] / z + rig.kl[3]], 1)
    pr = np.stack([rig.kr[0] * XR[:, 0] / XR[:, 2] + rig.kr[2], rig.kr[1] * XR[:, 1] / XR[:, 2] + rig.kr[3]], 1)
    pr += rng.normal(0, 0.4, pr.shape) + (rng.random((n, 1)) < 0.2) * rng.normal(0, 10.0, pr.shape)
    pl, pr = pl.astype(np.float32), pr.astype(np.float32)
    prm = S.GateParams(min_disp=1.0, z_min=3.0 * baseline, z_max=400.0 * baseline, max_reproj=1.5)
    r = S.stereo_gate(pl, pr, None, rig, prm)
    xyz, st, rs = _gpu_gate(pl, pr, None, rig, prm)
    bad = (rs != r.reason) & ~(r.margin < MARGIN)
    assert not bad.any(), (np.nonzero(bad)[0][:8], rs[bad][:8], r.reason[bad][:8], r.margin[bad][:8])
    assert (st == (rs == S.GATE_OK)).all()
    # the rows of each pair, for the bound
    L, Q = pl.astype(np.float64), pr.astype(np.float64)
    xl, yl = (L[:, 0] - rig.kl[2]) / rig.kl[0], (L[:, 1] - rig.kl[3]) / rig.kl[1]
    xr, yr = (Q[:, 0] - rig.kr[2]) / rig.kr[0], (Q[:, 1] - rig.kr[3]) / rig.kr[1]
    P = np.concatenate([R, rig.t[:, None]], 1)
    o, zr = np.ones(n), np.zeros(n)
    A = np.stack([np.stack([-o, zr, xl, zr], 1), np.stack([zr, -o, yl, zr], 1), xr[:, None] * P[2] - P[0],
                  yr[:, None] * P[2] - P[1]], 1)
    _, sv, vt = np.linalg.svd(A)
    x4 = np.abs(vt[:, 3, 3])
    ex = 64 * 2.0**-53 * sv[:, 0] ** 2 / (sv[:, 2] ** 2 - sv[:, 3] ** 2) + 1e-13
    X = r.xyz
    tol = 2.0**-24 * np.abs(X) + (ex * (1 + np.linalg.norm(X, axis=1)) / x4)[:, None]
    same = (rs == r.reason) & ((rs == S.GATE_OK) | (rs == S.GATE_DEPTH) | (rs == S.GATE_REPROJ))
    d = np.abs(xyz.astype(np.float64) - X)
    assert (d[same] <= tol[same]).all(), (d[same] / tol[same]).max()
    if n == 3000 and angle < 0.1:
        assert (rs == S.GATE_OK).sum() > 500
