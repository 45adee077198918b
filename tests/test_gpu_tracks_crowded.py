"""Carry-over of pools whose survivors crowd together, which are thinned one by
one instead of in rounds: the same decisions, at sizes around the step of 32 and
the CTA, and a time of the order of a spread-out pool's.  Compared for equality
with the greedy in priority order, single precision operation by operation."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

f32 = np.float32


def _greedy(pts, md):
    kept = np.zeros((0,), np.int64)
    for k in range(len(pts)):
        dx, dy = pts[k, 0] - pts[kept, 0], pts[k, 1] - pts[kept, 1]
        if not ((dx * dx + dy * dy) < f32(md) * f32(md)).any():
            kept = np.append(kept, k)
    return kept


def _layout(kind, m, rng):
    if kind == "same":
        return np.full((m, 2), 7.25)
    if kind == "cluster":
        return rng.normal(500, 25, (m, 2))
    if kind == "line":  # each conflicts with the two before it
        return np.stack([np.arange(m) * 4.5, np.zeros(m)], 1)
    if kind == "outlier":  # the grid's cells as wide as everything but one
        p = rng.uniform(0, 40 * np.sqrt(m), (m, 2))
        p[m // 2] = [1e7, 1e7]
        return p
    p = rng.uniform(0, 100 * np.sqrt(m), (m, 2))  # "pile": spread out, with five in one place
    p[rng.permutation(m)[:5]] = p[0] + 0.5
    p[m // 3] = [np.nan, 3.0]
    return p


def _pool(vt, torch, pts, ages):
    m = len(pts)
    p = vt.TrackPool(m)
    p.ids.copy_(torch.arange(m, dtype=torch.int32))
    p.ages.copy_(torch.from_numpy(ages))
    p.count.fill_(m)
    return p


@pytest.mark.parametrize("kind", ["same", "cluster", "line", "outlier", "pile"])
@pytest.mark.parametrize("ordered", [True, False])
def test_crowded(kind, ordered):
    import torch

    import paper_2607_01757_gb300 as vt

    md = 10.0
    for m in (2, 31, 32, 33, 64, 250, 1024, 1025, 4096):
        rng = np.random.Generator(np.random.PCG64(m))
        pts = _layout(kind, m, rng).astype(f32)
        ages = rng.integers(1, 6, m).astype(np.int32)
        if ordered:
            ages = np.ascontiguousarray(np.sort(ages)[::-1])
        order = np.argsort(-ages, kind="stable")
        want = order[_greedy(pts[order], md)]
        trk, st = torch.from_numpy(pts).cuda(), torch.ones(m, dtype=torch.uint8, device="cuda")
        for _ in range(3):
            p = _pool(vt, torch, pts, ages)
            vt.vt_tracks_carry([vt.carry_job(p, trk, st)], md)
            torch.cuda.synchronize()
            n = int(p.count.item())
            assert n == len(want), (m, n, len(want))
            assert np.array_equal(p.ids[:n].cpu().numpy(), want)
            assert np.array_equal(p.ages[:n].cpu().numpy(), ages[want] + 1)


def test_time():
    """A crowded pool takes no more than 50 times a spread-out one's time (settled
    in rounds, 4,096 survivors in one place took 1,000 times as long)."""
    import torch

    import paper_2607_01757_gb300 as vt

    m, us = 4096, {}
    rng = np.random.Generator(np.random.PCG64(1))
    for kind in ("pile", "same", "cluster"):
        pts = _layout(kind, m, rng).astype(f32)
        ages = np.full(m, 3, np.int32)
        trk, st = torch.from_numpy(pts).cuda(), torch.ones(m, dtype=torch.uint8, device="cuda")
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for _ in range(10):
            p = _pool(vt, torch, pts, ages)
            torch.cuda.synchronize()
            a.record()
            vt.vt_tracks_carry([vt.carry_job(p, trk, st)], 200.0)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3)
        us[kind] = best
    assert us["same"] < 50 * us["pile"] and us["cluster"] < 50 * us["pile"], us
