"""Carry-over and spawning at the edges of their launch: pool sizes around the
warp, the smallest and the largest CTA, in priority order (as a loop's own
pools are) and out of it, spread out, crowded (many closer neighbours) and in
a line (a chain of conflicts as long as the pool).  Compared for equality."""

import numpy as np
import pytest

from oracle import tracks as T

pytestmark = pytest.mark.gpu

SIZES = [1, 31, 33, 127, 128, 129, 255, 257, 1023, 1024, 1025, 2047]


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("caps", [SIZES[:5], SIZES, [4096]])
def test_carry_and_spawn_sizes(caps, ordered):
    import torch

    import paper_2607_01757_gb300 as vt

    rng = np.random.Generator(np.random.PCG64(len(caps) + 10 * ordered))
    md = 6.0
    pools, refs, jobs, masks, keep = [], [], [], [], []
    for cap in caps:
        for kind in ("spread", "crowd", "line") if cap <= 1025 else ("spread", "crowd"):
            n = cap if kind == "crowd" else max(1, cap - 3)
            if kind == "line":
                pts = np.stack([np.arange(n) * 5.0, np.full(n, 7.0)], 1)
            else:
                pts = rng.uniform(0, 30.0 if kind == "crowd" else 900.0 if cap <= 1025 else 150.0, (n, 2))
            ages = rng.integers(1, 9, n)
            if ordered:
                ages = np.sort(ages)[::-1]
            ref = T.Pool(pts.astype(np.float32), rng.permutation(5 * n).astype(np.int32)[:n],
                         ages.astype(np.int32), 10 ** 5)
            status = (rng.random(n) > (0.0 if kind == "line" else 0.1)).astype(np.uint8)
            p = vt.TrackPool(cap)
            p.pts[:n] = torch.from_numpy(ref.pts)
            p.ids[:n] = torch.from_numpy(ref.ids)
            p.ages[:n] = torch.from_numpy(np.ascontiguousarray(ref.ages))
            p.count[0] = n
            p.next_id[0] = ref.next_id
            tk, st = torch.from_numpy(ref.pts).cuda(), torch.from_numpy(status).cuda()
            mask = torch.zeros((cap, 2), device="cuda")
            jobs.append(vt.carry_job(p, tk, st, mask))
            pools.append(p)
            masks.append(mask)
            keep += [tk, st]
            refs.append((T.carry(ref, ref.pts, status, md), cap))
    vt.vt_tracks_carry(jobs, md)
    corners = torch.from_numpy(rng.uniform(0, 900, (1500, 2)).astype(np.float32)).cuda()
    cnt = torch.tensor([1500], dtype=torch.int32, device="cuda")
    kept = [p.count.clone() for p in pools]
    vt.vt_tracks_spawn([vt.spawn_job(p, corners, cnt) for p in pools])
    torch.cuda.synchronize()
    for p, (ref, cap), mask, k in zip(pools, refs, masks, kept):
        assert int(k.item()) == len(ref.ids)
        m = mask.cpu().numpy()
        assert np.array_equal(m[:len(ref.ids)], ref.pts) and np.isnan(m[len(ref.ids):]).all()
        ref = T.spawn(ref, corners.cpu().numpy(), None, cap)
        n = int(p.count.item())
        assert n == len(ref.ids) and int(p.next_id.item()) == ref.next_id
        assert np.array_equal(p.pts[:n].cpu().numpy(), ref.pts)
        assert np.array_equal(p.ids[:n].cpu().numpy(), ref.ids)
        assert np.array_equal(p.ages[:n].cpu().numpy(), ref.ages)
