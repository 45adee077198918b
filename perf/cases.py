"""What this library's users have it do, as cases that can be timed and checked.

The kinds of work, each through the package's public calls:

* ``pyramid``   one camera frame's image pyramid and gradient planes (vt_pyramid_build / _build_grad);
* ``track``     the points of one image pair, forward-backward or forward from a predicted position;
* ``streams``   one step of BatchedTracker: every stream's new frame(s) built, its points tracked to the new
                frame and, in stereo, from left to right, optionally with the triangulation gate;
* ``detect``    Shi-Tomasi corners of one or many frames away from points that are tracked already;
* ``gate``      the triangulation gate alone, on flow-checked stereo pairs;
* ``frontend``  one step of the whole device loop (tracking, bookkeeping, detection, cross-camera check, spawning).

Frames are seeded textures (blurred noise at several scales plus soft-edged patches) seen under small rigid
motions, with sensor noise; points are drawn on textured pixels at sub-pixel positions.
"""

from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2607_01757_gb300 as vt
from paper_2607_01757_gb300.engine import BatchedTracker
from paper_2607_01757_gb300.frontend import FrontEnd

DEV = "cuda"
GRADS = {"s16": vt.VT_GRAD_S16, "f16": vt.VT_GRAD_F16, "none": vt.VT_GRAD_NONE}
SHAPES = ((640, 480), (752, 480), (960, 600), (1440, 1080), (1920, 1200))


# ------------------------------------------------------------------------------- cases
def _pyramid(name, w, h, levels, grad="s16", host=False):
    return dict(name=name, kind="pyramid", w=w, h=h, levels=levels, grad=grad, host=host)


def _track(name, w, h, n, levels, win=21, grad="s16", fb=True):
    return dict(name=name, kind="track", w=w, h=h, n=n, levels=levels, win=win, grad=grad, fb=fb)


def _streams(name, streams, mix, gate=False, grad="s16", odd=False):
    return dict(name=name, kind="streams", streams=streams, mix=mix, gate=gate, grad=grad, odd=odd)


def _detect(name, frames, mix, corners, masked, min_dist=10, block=1, odd=False):
    return dict(name=name, kind="detect", frames=frames, mix=mix, corners=corners, masked=masked, min_dist=min_dist,
                block=block, odd=odd)


def listed():
    return [
        # a robot's single camera, frame by frame: the pyramid of one new frame ...
        _pyramid("pyramid-752x480", 752, 480, 4),
        # ... and one of a large sensor with odd sides, half-precision planes
        _pyramid("pyramid-1919x1199-f16", 1919, 1199, 6, grad="f16"),
        # the paper's pairing: 150 corners of one image pair with the forward-backward check; latency counts
        _track("track-752x480-150", 752, 480, 150, 4),
        # a learned extractor's density on a 1.3 MP sensor, half-precision planes
        _track("track-1280x1024-2000-f16", 1280, 1024, 2000, 5, grad="f16"),
        # odd frame, small window, predicted positions, no gradient planes kept
        _track("track-641x479-777-guess", 641, 479, 777, 4, win=15, grad="none", fb=False),
        # one camera served alone: the request a server gets at low load
        _streams("streams-1", 1, 12),
        # a small rig of cameras with the stereo gate
        _streams("streams-6-gate", 6, 4, gate=True),
        # the throughput workload: 32 cameras of uneven shapes
        _streams("streams-32", 32, 4),
        # new corners for one camera whose pool is half full
        _detect("detect-752x480", 1, 1, 256, 128),
        # new corners for 32 cameras in one call
        _detect("detect-32", 32, 4, 1000, 200),
        # stereo pairs of many cameras through the gate
        dict(name="gate-19000", kind="gate", n=19000),
        # the whole loop for eight cameras
        dict(name="frontend-8", kind="frontend", streams=8, mix=3, cap=256, odd=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pyramid", "pyramid", "track", "track", "streams", "streams", "detect", "gate", "frontend"])
    w = _log(rng, 320, 1920)
    h = max(240, min(1200, int(w * rng.uniform(0.55, 0.8))))
    mix = rng.randrange(1, 1 << 20)
    grad = rng.choice(["s16", "s16", "f16", "none"])
    if kind == "pyramid":
        c = _pyramid("", w, h, rng.randint(3, 6), grad=grad, host=rng.random() < 0.3)
    elif kind == "track":
        c = _track("", w, h, _log(rng, 50, 2000), rng.randint(3, 6), win=rng.choice([9, 15, 21, 21, 21, 31]), grad=grad,
                   fb=rng.random() < 0.7)
    elif kind == "streams":
        n = _log(rng, 1, 24)
        c = _streams("", n, mix, gate=n <= 12 and rng.random() < 0.5, grad=rng.choice(["s16", "s16", "s16", "f16"]),
                     odd=rng.random() < 0.5)
    elif kind == "detect":
        c = _detect("", _log(rng, 1, 16), mix, _log(rng, 100, 2000), rng.choice([0, 50, 200]), rng.choice([6, 10, 20]),
                    block=rng.choice([1, 1, 2]), odd=rng.random() < 0.5)
    elif kind == "gate":
        c = dict(kind="gate", n=_log(rng, 200, 19000))
    else:
        c = dict(kind="frontend", streams=_log(rng, 1, 12), mix=mix, cap=rng.choice([128, 200, 256, 500]),
                 odd=rng.random() < 0.5)
    c.pop("name", None)
    return c


def _specs(count, mix, odd):
    """Cameras of uneven shapes: mono or stereo, 200-2000 points, 4-6 levels; odd: sides a few pixels smaller."""
    r = random.Random(mix * 7919 + count)
    out = []
    for sid in range(count):
        w, h = r.choice(SHAPES)
        if odd:
            w, h = w - r.randrange(0, 8), h - r.randrange(0, 8)
        out.append(SimpleNamespace(sid=sid, w=w, h=h, stereo=r.random() < 0.5, n_kp=r.randint(200, 2000),
                                   levels=r.choice([4, 5, 6])))
    return out


# ------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _blur(a, sigma):
    r = int(math.ceil(2.5 * sigma))
    k = [math.exp(-0.5 * (i / sigma) ** 2) for i in range(-r, r + 1)]
    s = sum(k)
    for dim in (0, 1):
        acc = torch.zeros_like(a)
        for i, c in zip(range(-r, r + 1), k):
            acc += torch.roll(a, i, dim) * (c / s)
        a = acc
    return a


class _Scene:
    """A seeded texture with a margin around the w x h view, seen under rigid motions."""

    M = 64

    def __init__(self, w, h, g):
        self.w, self.h, self.g = w, h, g
        W, H = w + 2 * self.M, h + 2 * self.M
        t = torch.zeros((H, W), device=DEV)
        for sigma, amp in ((1.5, 9.0), (3.0, 16.0), (6.0, 22.0)):
            b = _blur(torch.randn((H, W), generator=g, device=DEV), sigma)
            t += b * (amp / (0.2821 / sigma))  # white noise blurred by sigma has deviation 1 / (2 sqrt(pi) sigma)
            if sigma == 6.0:
                t += 24.0 * torch.tanh(b * (4.0 / (0.2821 / sigma)))
        self.tex = (t + 128.0)[None, None]

    def view(self, theta_deg=0.0, tx=0.0, ty=0.0, shift=0.0, vshift=0.0):
        """uint8 [h, w]; a scene point at p in the unmoved view appears at R(theta)(p - c) + c + t - (shift, -vshift)."""
        w, h, M = self.w, self.h, self.M
        x = torch.arange(w, device=DEV, dtype=torch.float32)[None, :] + shift - tx - (w - 1) / 2
        y = torch.arange(h, device=DEV, dtype=torch.float32)[:, None] - vshift - ty - (h - 1) / 2
        c, s = math.cos(math.radians(theta_deg)), math.sin(math.radians(theta_deg))
        X = c * x + s * y + (w - 1) / 2 + M
        Y = -s * x + c * y + (h - 1) / 2 + M
        grid = torch.stack([X * (2.0 / (w + 2 * M - 1)) - 1.0, Y * (2.0 / (h + 2 * M - 1)) - 1.0], -1)[None]
        v = torch.nn.functional.grid_sample(self.tex, grid, mode="bicubic", padding_mode="reflection", align_corners=True)
        v = v[0, 0] + torch.randn((h, w), generator=self.g, device=DEV)
        return v.round().clamp(0, 255).to(torch.uint8).contiguous()


def _points(img, n, g, margin=24):
    """n textured sub-pixel positions of img, float32 [n, 2]."""
    f = img.float()
    h, w = img.shape
    dx, dy = torch.zeros_like(f), torch.zeros_like(f)
    dx[:, 1:-1] = (f[:, 2:] - f[:, :-2]) * 0.5
    dy[1:-1] = (f[2:] - f[:-2]) * 0.5

    def box(a):
        return torch.nn.functional.avg_pool2d(a[None, None], 7, 1, 3)[0, 0]

    a, b, c = box(dx * dx), box(dx * dy), box(dy * dy)
    s = (a + c) * 0.5 - (((a - c) * 0.5) ** 2 + b * b).sqrt()
    s = s[margin:h - margin, margin:w - margin]
    flat = s.reshape(-1)
    order = torch.sort(flat, descending=True, stable=True).indices[: max(n, int(0.3 * flat.numel()))]
    pick = order[torch.randperm(order.numel(), generator=g, device=DEV)[:n]]
    xy = torch.stack([pick % s.shape[1], pick // s.shape[1]], 1).float() + margin
    return (xy + torch.rand((n, 2), generator=g, device=DEV) - 0.5).contiguous()


def _frames(sp, seed):
    """Two consecutive frames of a camera: left images, right images (or None), points of each left image."""
    r = random.Random(seed * 1009 + sp.sid * 17 + sp.w)
    g = _gen(r.randrange(1 << 60))
    sc = _Scene(sp.w, sp.h, g)
    a, d = r.uniform(0, 2 * math.pi), r.uniform(2.0, 6.0)
    motion = [(0.0, 0.0, 0.0), (r.uniform(-0.5, 0.5), d * math.cos(a), d * math.sin(a))]
    disp, vmis = r.uniform(4.0, 24.0), r.uniform(-0.4, 0.4)
    left = [sc.view(*m) for m in motion]
    right = [sc.view(*m, shift=disp, vshift=vmis) if sp.stereo else None for m in motion]
    return SimpleNamespace(left=left, right=right, pts=[_points(i, sp.n_kp, g) for i in left], motion=motion[1])


def _rig(w, h):
    f = 460.0 * w / 752.0
    k = (f, f, (w - 1) / 2.0, (h - 1) / 2.0)
    return vt.StereoRig(kl=k, kr=k, t=(-0.11, 0.0, 0.0))


class _Plane:
    """Device memory of a pyramid as torch.as_tensor takes it; the tensor made of it keeps the pyramid alive."""

    def __init__(self, pyr, ptr, shape, strides, typestr):
        self.pyr = pyr
        self.__cuda_array_interface__ = dict(shape=shape, strides=strides, typestr=typestr, data=(ptr, False), version=3)


def _planes(p, levels, grad):
    """Tensors over a built pyramid's images and gradient planes."""
    out = []
    for l in range(levels):
        ptr, w, h, pitch = vt.vt_pyramid_level(p, l)
        out.append(torch.as_tensor(_Plane(p, ptr, (h, w), (pitch, 1), "|u1"), device=DEV))
    for l in range(levels if grad != "none" else 0):
        ptr, pitch, _ = vt.vt_pyramid_grad(p, l)
        _, w, h, _ = vt.vt_pyramid_level(p, l)
        out.append(torch.as_tensor(_Plane(p, ptr, (h, w, 2), (4 * pitch, 4, 2), "<i2" if grad == "s16" else "<f2"), device=DEV))
    return out


def _build(img, levels, grad, out=None):
    if grad == "none":
        return vt.vt_pyramid_build(img, levels, out=out)
    return vt.vt_pyramid_build_grad(img, levels, GRADS[grad], out=out)


def _pair(c, seed):
    sp = SimpleNamespace(sid=0, w=c["w"], h=c["h"], stereo=False, n_kp=c["n"])
    f = _frames(sp, seed)
    th, tx, ty = f.motion
    p = f.pts[0].double()
    ctr = torch.tensor([(c["w"] - 1) / 2, (c["h"] - 1) / 2], device=DEV, dtype=torch.float64)
    cs, sn = math.cos(math.radians(th)), math.sin(math.radians(th))
    R = torch.tensor([[cs, -sn], [sn, cs]], device=DEV, dtype=torch.float64)
    true = (p - ctr) @ R.T + ctr + torch.tensor([tx, ty], device=DEV, dtype=torch.float64)
    f.guess = (true + (torch.rand(p.shape, generator=_gen(seed * 31 + 5), device=DEV) - 0.5) * 4.0).float().contiguous()
    return f


def _detect_inputs(c, seed):
    out = []
    for sp in _specs(c["frames"], c["mix"], c["odd"]):
        f = _frames(SimpleNamespace(sid=sp.sid, w=sp.w, h=sp.h, stereo=False, n_kp=max(1, c["masked"])), seed)
        out.append((sp, f.left[0], f.pts[0] if c["masked"] else None))
    return out


def _gate_inputs(c, seed):
    """Pairs as the flow check leaves them: points in front of the rig with pixel noise, some too far, some mistracked."""
    g = np.random.Generator(np.random.PCG64(seed))
    n = c["n"]
    rot = g.normal(0, 0.01, 3)
    K = np.array([[0, -rot[2], rot[1]], [rot[2], 0, -rot[0]], [-rot[1], rot[0], 0]])
    th = np.linalg.norm(rot)
    R = np.eye(3) + np.sin(th) / th * K + (1 - np.cos(th)) / th**2 * (K @ K)
    kl, kr = (458.7, 457.3, 367.2, 248.4), (457.6, 456.1, 379.9, 255.2)
    t = np.array([-0.11, 0.001, -0.002])
    Z = np.exp(g.uniform(np.log(0.5), np.log(60.0), n))
    ul, vl = g.uniform(0, 751, n), g.uniform(0, 479, n)
    X = np.stack([(ul - kl[2]) / kl[0] * Z, (vl - kl[3]) / kl[1] * Z, Z], 1)
    Y = X @ R.T + t
    pr = np.stack([kr[0] * Y[:, 0] / Y[:, 2] + kr[2], kr[1] * Y[:, 1] / Y[:, 2] + kr[3]], 1)
    pr += g.normal(0, 0.3, pr.shape) + (g.random((n, 1)) < 0.05) * g.normal(0, 8.0, pr.shape)
    st = (g.random(n) < 0.92).astype(np.uint8)
    return np.stack([ul, vl], 1).astype(np.float32), pr.astype(np.float32), st, (kl, kr, R, t)


# ------------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    return {"pyramid": _prep_pyramid, "track": _prep_track, "streams": _prep_streams, "detect": _prep_detect,
            "gate": _prep_gate, "frontend": _prep_frontend}[case["kind"]](case, seed)


def run(s):
    return s.go()


def _prep_pyramid(c, seed):
    img = _pair(dict(c, n=1), seed).left[0]
    if c["host"]:
        img = img.cpu().pin_memory()
    pyr = vt.vt_pyramid_create(c["w"], c["h"], c["levels"])
    _build(img, c["levels"], c["grad"], pyr)
    planes = _planes(pyr, c["levels"], c["grad"])

    def go():
        _build(img, c["levels"], c["grad"], pyr)
        return planes

    return SimpleNamespace(go=go, keep=(img, pyr))


def _prep_track(c, seed):
    f = _pair(c, seed)
    I, J = (_build(i, c["levels"], c["grad"]) for i in f.left)
    prm = vt.KltParams(win=c["win"], levels=c["levels"])
    out = torch.zeros((c["n"], 2), device=DEV)
    st = torch.zeros(c["n"], dtype=torch.uint8, device=DEV)
    err = torch.zeros(c["n"], device=DEV)

    def go():
        if c["fb"]:
            vt.vt_klt_track_fb(I, J, f.pts[0], prm, out, st, err)
        else:
            vt.vt_klt_track_ex(I, J, f.pts[0], prm, out, st, err, pts_guess=f.guess)
        return out, st, err

    return SimpleNamespace(go=go, keep=(I, J, f))


def _prep_streams(c, seed):
    specs = _specs(c["streams"], c["mix"], c["odd"])
    fr = [_frames(sp, seed) for sp in specs]
    tr = BatchedTracker(specs, vt.KltParams(levels=4), grad_type=GRADS[c["grad"]],
                        gate=vt.GateParams() if c["gate"] else None,
                        rigs=[_rig(sp.w, sp.h) if sp.stereo else None for sp in specs] if c["gate"] else None)
    sids = list(range(len(specs)))
    n = [sp.n_kp for sp in specs]
    zero = [0] * len(specs)
    step = [0]

    def frame(track):
        k = step[0] % 2
        tr.stage(tr.step_tables(sids, n if track else zero, n if track else zero, left=[f.left[k] for f in fr],
                                right=[f.right[k] for f in fr], kpt=[f.pts[1 - k] for f in fr],
                                kps=[f.pts[k] for f in fr]))
        tr.run()
        tr.advance(sids)
        step[0] += 1

    frame(False)
    frame(False)
    # the first camera's planes after a step, for either of its two pyramids
    planes = [_planes(p, specs[0].levels, c["grad"]) for p in tr.streams[0].pyr]
    gates = [s.gate_out for s in tr.streams if s.rig is not None]

    def go():
        frame(True)
        return tr.out_pts, tr.out_st, tr.out_err, tr.out_rs, gates, planes[tr.streams[0].built % 2]

    return SimpleNamespace(go=go, keep=(tr, fr))


def _prep_detect(c, seed):
    jobs, keep = [], []
    inputs = _detect_inputs(c, seed)
    cap = c["corners"]
    xy = torch.zeros((len(inputs), cap, 2), device=DEV)
    sc = torch.zeros((len(inputs), cap), device=DEV)
    cnt = torch.zeros(len(inputs), dtype=torch.int32, device=DEV)
    prm = vt.GfttParams(max_corners=cap, quality=0.01, min_dist=c["min_dist"], nms_radius=4, block_radius=c["block"],
                        border=10)
    for k, (sp, img, mask) in enumerate(inputs):
        p = _build(img, 1, "s16")
        jobs.append(vt.gftt_job(p, 0, xy[k], cnt[k:k + 1], cap, scores_out=sc[k], mask=mask))
        keep.append((p, mask))
    g = vt.vt_gftt_create_pixels(sum(sp.w * sp.h for sp, _, _ in inputs))

    def go():
        if len(jobs) == 1:
            vt.vt_gftt_detect(g, keep[0][0], 0, prm, xy[0], cnt, sc[0], mask=keep[0][1])
        else:
            vt.vt_gftt_detect_many(g, jobs, prm)
        return xy, sc, cnt

    return SimpleNamespace(go=go, keep=(keep, g))


def _prep_gate(c, seed):
    pl, pr, st, (kl, kr, R, t) = _gate_inputs(c, seed)
    pl, pr, st = (torch.from_numpy(a).to(DEV) for a in (pl, pr, st))
    rig, prm = vt.StereoRig(kl, kr, R, t), vt.GateParams()
    ok = torch.zeros(c["n"], dtype=torch.uint8, device=DEV)
    why = torch.zeros(c["n"], dtype=torch.uint8, device=DEV)
    xyz = torch.zeros((c["n"], 3), device=DEV)

    def go():
        vt.vt_stereo_gate(pl, pr, rig, prm, ok, status_in=st, xyz_out=xyz, reason_out=why)
        return ok, xyz, why

    return SimpleNamespace(go=go)


def _prep_frontend(c, seed):
    specs = _specs(c["streams"], c["mix"], c["odd"])
    fr = [_frames(SimpleNamespace(sid=sp.sid, w=sp.w, h=sp.h, stereo=sp.stereo, n_kp=1), seed) for sp in specs]
    fe = FrontEnd(specs, vt.KltParams(levels=4), cap=c["cap"])
    step = [0]

    def go():
        k = step[0] % 2
        fe.step([f.left[k] for f in fr], [f.right[k] for f in fr])
        step[0] += 1
        return [(d["pool"].pts, d["pool"].ids, d["pool"].ages, d["pool"].count) for d in fe.st]

    go()
    return SimpleNamespace(go=go, keep=(fe, fr))


# ------------------------------------------------------------------------------- work
def _pyr_px(w, h, levels):
    px = 0
    for _ in range(levels):
        px += w * h
        w, h = (w + 1) // 2, (h + 1) // 2
    return px


def _pyr_work(w, h, levels, grad):
    px = _pyr_px(w, h, levels)
    up = px - w * h  # pixels of the levels above 0; level 0 is read once and kept
    return dict(bytes=2 * w * h + up + (0 if grad == "none" else 4 * px), flops=(0 if grad == "none" else 16 * px) + 18 * up)


def _track_work(n, win, levels, passes, w, h, grad):
    # per pass: a template sweep (27 per sample) and about three Newton iterations (12) a level, the first pass's
    # error sweep (9); the windows of both frames, and no more than the frames hold
    s = win * win
    px = _pyr_px(w, h, levels)
    b = 1 if grad == "none" else 5
    return dict(bytes=min(n * levels * passes * (win + 1) ** 2 * (b + 1), 2 * px * b) + n * (8 + 8 + 1 + 4),
                flops=n * s * (passes * levels * (27 + 3 * 12) + 9))


def _gate_work(n):
    return dict(bytes=n * (17 + 14), flops=n * 2000)


def _detect_work(w, h, block, corners, masked):
    # box sums of three products (separable), the score, the window maximum
    return dict(bytes=4 * w * h + 12 * corners + 8 * masked, flops=w * h * (3 + 6 * 2 * block + 9 + 16))


def work(case):
    c, k = case, case["kind"]
    parts = []
    if k == "pyramid":
        parts = [_pyr_work(c["w"], c["h"], c["levels"], c["grad"])]
    elif k == "track":
        parts = [_track_work(c["n"], c["win"], c["levels"], 2 if c["fb"] else 1, c["w"], c["h"], c["grad"])]
    elif k == "streams":
        for sp in _specs(c["streams"], c["mix"], c["odd"]):
            for _ in range(2 if sp.stereo else 1):
                parts += [_pyr_work(sp.w, sp.h, sp.levels, c["grad"]),
                          _track_work(sp.n_kp, 21, sp.levels, 2, sp.w, sp.h, c["grad"])]
            if c["gate"] and sp.stereo:
                parts += [_gate_work(sp.n_kp)]
    elif k == "detect":
        for sp in _specs(c["frames"], c["mix"], c["odd"]):
            parts += [_detect_work(sp.w, sp.h, c["block"], c["corners"], c["masked"])]
    elif k == "gate":
        parts = [_gate_work(c["n"])]
    else:
        for sp in _specs(c["streams"], c["mix"], c["odd"]):
            parts += [_pyr_work(sp.w, sp.h, sp.levels, "s16")] * (2 if sp.stereo else 1)
            parts += [_track_work(c["cap"], 21, sp.levels, 2, sp.w, sp.h, "s16"),
                      _detect_work(sp.w, sp.h, 1, c["cap"], c["cap"])]
            if sp.stereo:
                parts += [_track_work(c["cap"], 21, sp.levels, 2, sp.w, sp.h, "s16")]
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


# ------------------------------------------------------------------------------- the same in 64 bits
def _refl(n, r):
    """Indices -r .. n-1+r reflected into 0 .. n-1 without repeating the edge (a side of 1 clamps)."""
    i = np.arange(-r, n + r)
    if n == 1:
        i[:] = 0
    while n > 1 and ((i < 0) | (i >= n)).any():
        i = np.where(i < 0, -i, i)
        i = np.where(i >= n, 2 * n - 2 - i, i)
    return torch.from_numpy(i).to(DEV)


def _pad(a, r):
    return a[_refl(a.shape[0], r)][:, _refl(a.shape[1], r)]


def _pyr64(img, levels):
    out = [img.to(DEV).to(torch.int64)]
    for _ in range(levels - 1):
        a = out[-1]
        H, W = (a.shape[0] + 1) // 2, (a.shape[1] + 1) // 2
        p = _pad(a, 2)
        v = sum(k * p[i:i + 2 * H - 1:2] for i, k in enumerate((1, 4, 6, 4, 1)))
        s = sum(k * v[:, i:i + 2 * W - 1:2] for i, k in enumerate((1, 4, 6, 4, 1)))
        out.append((s + 128) >> 8)
    return out


def _scharr64(a):
    p = _pad(a, 1)
    d, s = p[:, 2:] - p[:, :-2], p[2:] - p[:-2]
    return 3 * (d[:-2] + d[2:]) + 10 * d[1:-1], 3 * (s[:, :-2] + s[:, 2:]) + 10 * s[:, 1:-1]


def _planes64(img, levels, grad):
    py = _pyr64(img, levels)
    out = list(py)
    if grad != "none":
        for a in py:
            g = torch.stack(_scharr64(a), -1)
            out.append(g if grad == "s16" else g.double() / 32.0)
    return out


def _bilinear(a, x, y):
    h, w = a.shape
    fx, fy = x.floor(), y.floor()
    bx, by = x - fx, y - fy
    x0, y0 = fx.long().clamp(0, w - 1), fy.long().clamp(0, h - 1)
    x1, y1 = (fx.long() + 1).clamp(0, w - 1), (fy.long() + 1).clamp(0, h - 1)
    f = a.reshape(-1)
    p, q = f[y0 * w + x0], f[y0 * w + x1]
    top = p + bx * (q - p)
    p, q = f[y1 * w + x0], f[y1 * w + x1]
    return top + by * (p + bx * (q - p) - top)


def _track64(I, J, pts, win, guess=None, iters=30, eps=0.01, min_eig=1e-4):
    """Coarse-to-fine Lucas-Kanade of pts from pyramid I to pyramid J: positions, status, mean |T - J|."""
    hw = win // 2
    o = torch.arange(-hw, hw + 1, device=DEV, dtype=torch.float64)
    ox, oy = o.repeat(win)[None], o.repeat_interleave(win)[None]
    n, L = pts.shape[0], len(I)
    ok = (pts[:, 0] >= 0) & (pts[:, 0] <= I[0].shape[1] - 1) & (pts[:, 1] >= 0) & (pts[:, 1] <= I[0].shape[0] - 1)
    g = torch.zeros_like(pts) if guess is None else (guess - pts) / 2 ** (L - 1)
    res, err = pts.clone(), torch.zeros(n, device=DEV, dtype=torch.float64)
    for l in range(L - 1, -1, -1):
        a, b = I[l].double(), J[l].double()
        gx, gy = (t.double() / 32.0 for t in _scharr64(I[l]))
        at = ok.nonzero()[:, 0]
        u = pts[at] / 2 ** l
        T, X, Y = (_bilinear(p, u[:, :1] + ox, u[:, 1:] + oy) for p in (a, gx, gy))
        A, B, C = (X * X).sum(1), (X * Y).sum(1), (Y * Y).sum(1)
        det = A * C - B * B
        lmin = ((A + C) - ((A - C) ** 2 + 4 * B * B).sqrt()) / 2 / (win * win * 65025.0)
        good = (lmin >= min_eig) & (det > 0)
        nu = torch.zeros_like(u)
        oob = torch.zeros_like(good)
        act = good.nonzero()[:, 0]
        h, w = b.shape
        for _ in range(iters):
            if not act.numel():
                break
            q = u[act] + g[at[act]] + nu[act]
            inside = ((q >= -hw) & (q <= torch.tensor([w - 1 + hw, h - 1 + hw], device=DEV))).all(1)
            oob[act[~inside]] = True
            act, q = act[inside], q[inside]
            r = T[act] - _bilinear(b, q[:, :1] + ox, q[:, 1:] + oy)
            b1, b2 = (r * X[act]).sum(1), (r * Y[act]).sum(1)
            e = torch.stack([C[act] * b1 - B[act] * b2, A[act] * b2 - B[act] * b1], 1) / det[act][:, None]
            nu[act] += e
            act = act[(e * e).sum(1) >= eps * eps]
        lost = ~good | oob
        res[at] = (u + g[at] + nu) * 2 ** l
        ok[at[lost]] = False
        if l > 0:
            g[at] = torch.where(lost[:, None], g[at], 2 * (g[at] + nu))
        else:
            p = res[at]
            out = ~((p >= 0) & (p <= torch.tensor([w - 1, h - 1], device=DEV))).all(1)
            ok[at[out]] = False
            e = (T - _bilinear(b, p[:, :1] + ox, p[:, 1:] + oy)).abs().mean(1)
            err[at] = torch.where(out | lost, torch.zeros_like(e), e)
    return res, ok, err


def _track_fb64(I, J, pts, win, thr=0.5):
    """The forward pass, and the status after the backward pass from its result."""
    p, ok, err = _track64(I, J, pts, win)
    at = ok.nonzero()[:, 0]
    back, okb, _ = _track64(J, I, p[at], win)
    ok[at] = okb & (((back - pts[at]) ** 2).sum(1) <= thr * thr)
    return p, ok, torch.where(ok, err, torch.zeros_like(err))


def _gate64(pl, pr, st, rig):
    """Status, points and reasons of the triangulation gate (min_disp 1, depth 0.1 to 50, reprojection 1.5)."""
    kl, kr, R, t = (np.asarray(v, np.float64) for v in rig)
    R = R.reshape(3, 3)
    pl, pr = pl.astype(np.float64), pr.astype(np.float64)
    xl, yl = (pl[:, 0] - kl[2]) / kl[0], (pl[:, 1] - kl[3]) / kl[1]
    xr, yr = (pr[:, 0] - kr[2]) / kr[0], (pr[:, 1] - kr[3]) / kr[1]
    ray = np.stack([xl, yl, np.ones_like(xl)], 1) @ R.T
    with np.errstate(all="ignore"):
        d = np.hypot(pr[:, 0] - (kr[0] * ray[:, 0] / ray[:, 2] + kr[2]), pr[:, 1] - (kr[1] * ray[:, 1] / ray[:, 2] + kr[3]))
        z, o = np.zeros_like(xl), np.ones_like(xl)
        P = np.concatenate([R, t[:, None]], 1)
        A = np.stack([np.stack([-o, z, xl, z], 1), np.stack([z, -o, yl, z], 1), xr[:, None] * P[2] - P[0],
                      yr[:, None] * P[2] - P[1]], 1)
        X = np.linalg.svd(A)[2][:, 3]
        X = X[:, :3] / X[:, 3:]
        Y = X @ R.T + t
        depth = (Y[:, 2] > 0) & (X[:, 2] >= 0.1) & (X[:, 2] <= 50.0)
        el = np.hypot(kl[0] * X[:, 0] / X[:, 2] + kl[2] - pl[:, 0], kl[1] * X[:, 1] / X[:, 2] + kl[3] - pl[:, 1])
        er = np.hypot(kr[0] * Y[:, 0] / Y[:, 2] + kr[2] - pr[:, 0], kr[1] * Y[:, 1] / Y[:, 2] + kr[3] - pr[:, 1])
    why = np.select([st == 0, (ray[:, 2] > 0) & ~(d > 1.0), ~depth, ~(np.maximum(el, er) <= 1.5)],
                    [vt.VT_LOST_INPUT, vt.VT_LOST_DISP, vt.VT_LOST_DEPTH, vt.VT_LOST_REPROJ], vt.VT_TRACKED)
    X[(why == vt.VT_LOST_INPUT) | (why == vt.VT_LOST_DISP)] = 0.0
    return (why == vt.VT_TRACKED).astype(np.uint8), X, why.astype(np.uint8)


def _thin(xy, order, min_dist, cap):
    """Greedy minimum-distance selection of xy[order], at most cap of them (None: all that are kept)."""
    cells, kept = {}, []
    for i in order:
        x, y = xy[i]
        cx, cy = int(x // min_dist), int(y // min_dist)
        near = (q for a in (-1, 0, 1) for b in (-1, 0, 1) for q in cells.get((cx + a, cy + b), ()))
        if any((x - q[0]) ** 2 + (y - q[1]) ** 2 < min_dist * min_dist for q in near):
            continue
        cells.setdefault((cx, cy), []).append((x, y))
        kept.append(i)
        if len(kept) == cap:
            break
    return kept


def _detect64(img, cap, min_dist, mask, block=1, nms=4, quality=0.01, border=10):
    """(corners [k, 2], scores [k]) of the Shi-Tomasi rules with scores in 64 bits."""
    gx, gy = _scharr64(_pyr64(img, 1)[0])
    h, w = gx.shape
    prod = [_pad(p, 0) for p in (gx * gx, gx * gy, gy * gy)]
    a, b, c = (sum(_pad(p, block)[j:j + h, i:i + w] for j in range(2 * block + 1) for i in range(2 * block + 1)).double()
               for p in prod)
    s = (((a + c) - ((a - c) ** 2 + 4 * b * b).sqrt()) / 2).clamp(min=0)
    ninf = float("-inf")
    top = torch.nn.functional.max_pool2d(s[None, None], 2 * nms + 1, 1, nms)[0, 0]
    cand = (s == top) & (s > 0) & (s >= quality * s.max())
    inner = torch.zeros_like(cand)
    inner[border:h - border, border:w - border] = True
    y, x = (cand & inner).nonzero(as_tuple=True)
    p = torch.nn.functional.pad(s, (nms,) * 4, value=ninf)
    for j in range(-nms, 1):
        for i in range(-nms, nms + 1):
            if j == 0 and i >= 0:
                break
            keep = p[y + nms + j, x + nms + i] < s[y, x]  # an equal score at a smaller index comes first
            y, x = y[keep], x[keep]
    if mask is not None and mask.numel():
        m = mask.double()[torch.isfinite(mask).all(1)]
        d2 = (x.double()[:, None] - m[:, 0]) ** 2 + (y.double()[:, None] - m[:, 1]) ** 2
        keep = ~(d2 < min_dist * min_dist).any(1)
        y, x = y[keep], x[keep]
    sc = s[y, x].cpu().numpy()
    xy = torch.stack([x, y], 1).cpu().numpy().astype(np.float64)
    kept = _thin(xy.tolist(), np.lexsort((xy[:, 1] * w + xy[:, 0], -sc)).tolist(), min_dist, cap) if cap else []
    return xy[kept].reshape(-1, 2), sc[kept]


def _streams64(c, seed):
    specs = _specs(c["streams"], c["mix"], c["odd"])
    pts, st, err, gates, planes = [], [], [], [], None
    for sp in specs:
        f = _frames(sp, seed)
        py = [_pyr64(i, sp.levels) for i in f.left]
        # the first pass after preparing: frame 0 arrives again, frame 1 is the previous one
        p, ok, e = _track_fb64(py[1], py[0], f.pts[1].double(), 21)
        pts, st, err = pts + [p], st + [ok], err + [e]
        if sp.stereo:
            q, ok, e = _track_fb64(py[0], _pyr64(f.right[0], sp.levels), f.pts[0].double(), 21)
            pts, st, err = pts + [q], st + [ok], err + [e]
            if c["gate"]:
                r = _rig(sp.w, sp.h)
                g = _gate64(f.pts[0].cpu().numpy(), q.cpu().numpy(), ok.cpu().numpy().astype(np.uint8), (r.kl, r.kr, r.R, r.t))
                gates.append((None, g[1], None))
        if planes is None:
            planes = _planes64(f.left[0], sp.levels, c["grad"])
    return torch.cat(pts), torch.cat(st).to(torch.uint8), torch.cat(err), None, gates, planes


def _frontend64(c, seed):
    out, cap, md = [], c["cap"], 10.0
    for sp in _specs(c["streams"], c["mix"], c["odd"]):
        f = _frames(SimpleNamespace(sid=sp.sid, w=sp.w, h=sp.h, stereo=sp.stereo, n_kp=1), seed)
        py = [_pyr64(i, sp.levels) for i in f.left]
        buf = np.zeros((cap, 2))
        pool = np.zeros((0, 2))
        for k in (0, 1):
            if k:  # every track is one frame old: priority is pool order
                p, ok, _ = _track_fb64(py[0], py[1], torch.from_numpy(pool).to(DEV), 21)
                p = p[ok].cpu().numpy()
                pool = p[_thin(p.tolist(), range(len(p)), md, None)].reshape(-1, 2)
                buf[:len(pool)] = pool
            xy, _ = _detect64(f.left[k], cap, 10, torch.from_numpy(pool).to(DEV))
            if sp.stereo and len(xy):
                _, ok, _ = _track_fb64(py[k], _pyr64(f.right[k], sp.levels), torch.from_numpy(xy).to(DEV), 21)
                xy = xy[ok.cpu().numpy()]
            pool = np.concatenate([pool, xy])[:cap]
            buf[:len(pool)] = pool
        out.append((buf, None, None, None))
    return out


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "pyramid":
        return _planes64(_pair(dict(c, n=1), seed).left[0], c["levels"], c["grad"])
    if k == "track":
        f = _pair(c, seed)
        I, J = (_pyr64(i, c["levels"]) for i in f.left)
        if c["fb"]:
            p, ok, err = _track_fb64(I, J, f.pts[0].double(), c["win"])
        else:
            p, ok, err = _track64(I, J, f.pts[0].double(), c["win"], guess=f.guess.double())
        return p, ok.to(torch.uint8), err
    if k == "streams":
        return _streams64(c, seed)
    if k == "detect":
        inputs = _detect_inputs(c, seed)
        xy = np.zeros((len(inputs), c["corners"], 2))
        sc = np.zeros((len(inputs), c["corners"]))
        cnt = np.zeros(len(inputs), np.int32)
        for i, (_, img, mask) in enumerate(inputs):
            p, s = _detect64(img, c["corners"], c["min_dist"], mask, c["block"])
            xy[i, :len(p)], sc[i, :len(p)], cnt[i] = p, s, len(p)
        return xy, sc, cnt
    if k == "gate":
        pl, pr, st, rig = _gate_inputs(c, seed)
        return _gate64(pl, pr, st, rig)
    return _frontend64(c, seed)
