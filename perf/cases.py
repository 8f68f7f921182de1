"""Workloads of the stereo visual frontend, as a user's program runs them.

Every case goes through the package's public calls on device-resident inputs:

  frame    vio.Frontend over a stereo sequence (a session in progress)
  batch    one vio.Batch step of stereo streams of mixed sizes
  detect   pyramid and grid detection of a set of images
  track    temporal tracking of keypoints between image pairs
  rig      one camera's keypoints matched into the other cameras of a rig,
           from the model-based start
  propose  the flow network's inputs and proposals of tracked keypoints
  train    one optimiser step of the flow network

Images are seeded stand-ins for camera frames: band-limited noise texture
(uniform noise, Gaussian of 2 px, mean 128, standard deviation 40) seen under
small SE(2) motion and scale, with N(0, 2^2) sensor noise, as uint8.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch
import torch.nn.functional as nnf

from paper_2609_30459_gb300 import vio

DEV = "cuda"
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(vio.__file__)), "data", "initnet.npz")


def listed():
    return [
        # one frame at a time at the cheapest setting (large cells, high
        # threshold, few iterations): the latency a small robot's loop sees
        dict(name="frame_lite", kind="frame", w=752, h=480, streams=1, levels=4, cw=82, ch=82,
             k=1, tmin=20, iters=3, steps=2, piped=False, learned=False, motion=15.0),
        # a recorded 752x480 stereo sequence played through the frontend, 300
        # cells: the usual offline and headline workload
        dict(name="frame_752x480", kind="frame", w=752, h=480, streams=1, levels=4, cw=37, ch=32,
             k=1, tmin=5, iters=5, steps=8, piped=True, learned=False, motion=15.0),
        # two 1920x1080 stereo pairs on one vehicle, 1000 cells each
        dict(name="frame_1080p_rig", kind="frame", w=1920, h=1080, streams=2, levels=5, cw=48,
             ch=43, k=1, tmin=5, iters=5, steps=4, piped=True, learned=False, motion=40.0),
        # a server's step: 16 streams of four sizes, learned start, replayed graph
        dict(name="batch_16_learned", kind="batch", learned=True, graph=True, motion=40.0,
             groups="640x480x4/32x32 752x480x4/37x32 1280x720x4/42x36 1920x1080x4/48x43",
             levels=5),
        # keypoints of one stereo pair: the smallest detection call
        dict(name="detect_pair", kind="detect", w=752, h=480, n=2, levels=4, cw=37, ch=32, k=1,
             tmin=5, select=0, rnd=0, mask=False, occ=False, fused=True),
        # a recorded sequence preprocessed in one call (larger than the L2)
        dict(name="detect_512", kind="detect", w=752, h=480, n=512, levels=4, cw=37, ch=32, k=1,
             tmin=5, select=0, rnd=0, mask=False, occ=False, fused=True),
        # separate stage calls with every option: odd size, several keypoints
        # per cell, a pixel mask (the robot's own body), occupied cells
        dict(name="detect_masked", kind="detect", w=641, h=479, n=12, levels=4, cw=50, ch=50, k=4,
             tmin=5, select=1, rnd=1, mask=True, occ=True, fused=False),
        # one image pair's keypoints: the smallest tracking call
        dict(name="track_pair", kind="track", w=752, h=480, pairs=1, cw=37, ch=32, levels=4,
             iters=5, fb=True, start=-1, motion=15.0),
        # every pair of a 21-frame sequence with 16-px cells (how the flow
        # network's training targets are made)
        dict(name="track_20_pairs", kind="track", w=640, h=480, pairs=20, cw=16, ch=16, levels=5,
             iters=5, fb=True, start=-1, motion=40.0),
        # a four-camera rig: 1000 keypoints into three cameras, from predictions
        dict(name="rig_1080p", kind="rig", w=1920, h=1080, targets=3, cw=48, ch=43, levels=5,
             iters=5),
        # proposals for the keypoints of 20 image pairs
        dict(name="propose_20_pairs", kind="propose", w=640, h=480, pairs=20, cw=16, ch=16,
             levels=5, la=2, lb=3, motion=40.0),
        # one minibatch of the flow network's training
        dict(name="train_1024", kind="train", n=1024, pool=8192, radius=3.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, wmax=1920, hmax=1080):
    """Image size, over the range of the listed ones, any parity."""
    w = _log(rng, 320, wmax)
    h = min(hmax, max(200, int(w * rng.uniform(0.5, 0.8))))
    return w, h


def _levels(rng, w, h, lo=3, hi=5):
    return min(rng.randint(lo, hi), int(math.log2(min(w, h) / 24.0)) + 1)


def _cell(rng, lo, hi):
    c = _log(rng, lo, hi)
    return c, max(lo, c - rng.randint(0, max(1, c // 6)))


def draw(rng):
    kind = rng.choice(["frame", "frame", "batch", "detect", "detect", "track", "track", "rig",
                       "propose", "train"])
    if kind == "frame":
        w, h = _size(rng)
        cw, ch = _cell(rng, 30, 82)
        streams = rng.choice([1, 1, 2])
        return dict(kind=kind, w=w, h=h, streams=streams, levels=_levels(rng, w, h), cw=cw, ch=ch,
                    k=rng.choice([1, 1, 2]), tmin=rng.choice([5, 5, 10, 20]),
                    iters=rng.choice([3, 5, 5]), steps=rng.choice([2, 4]),
                    piped=rng.random() < 0.5, learned=rng.random() < 0.3,
                    motion=round(rng.uniform(3.0, 40.0), 2))
    if kind == "batch":
        groups = []
        for _ in range(rng.randint(1, 4)):
            w, h = _size(rng)
            cw, ch = _cell(rng, 32, 60)
            groups.append("%dx%dx%d/%dx%d" % (w, h, rng.randint(1, 4), cw, ch))
        return dict(kind=kind, learned=rng.random() < 0.6, graph=rng.random() < 0.7,
                    motion=round(rng.uniform(3.0, 40.0), 2), groups=" ".join(groups), levels=4)
    if kind == "detect":
        w, h = _size(rng)
        n = max(1, min(_log(rng, 1, 512), 512 * 752 * 480 // (w * h)))
        cw, ch = _cell(rng, 8, 82)
        cells = n * (w // cw) * (h // ch)
        k = rng.choice([1, 1, 2, 4]) if cells < 100_000 else 1
        if cells > 160_000:
            n = max(1, n * 160_000 // cells)
        return dict(kind=kind, w=w, h=h, n=n, levels=_levels(rng, w, h, 1, 5), cw=cw, ch=ch, k=k,
                    tmin=rng.choice([5, 5, 10, 20]),
                    select=rng.choice([0, 0, 1, 2]) if k == 1 else rng.choice([0, 1]),
                    rnd=rng.choice([0, 0, 1]), mask=rng.random() < 0.3, occ=rng.random() < 0.4,
                    fused=rng.random() < 0.6)
    if kind in ("track", "propose"):
        w, h = _size(rng)
        cw, ch = _cell(rng, 16, 60)
        per = (w // cw) * (h // ch)
        pairs = max(1, min(_log(rng, 1, 20), 24_000 // per))
        levels = max(4, _levels(rng, w, h))
        motion = round(rng.uniform(3.0, 40.0), 2)
        if kind == "propose":
            return dict(kind=kind, w=w, h=h, pairs=pairs, cw=cw, ch=ch, levels=levels, la=2, lb=3,
                        motion=motion)
        return dict(kind=kind, w=w, h=h, pairs=pairs, cw=cw, ch=ch, levels=levels,
                    iters=rng.choice([3, 5, 5]), fb=rng.random() < 0.8,
                    start=rng.choice([-1, -1, 0, 1]), motion=motion)
    if kind == "rig":
        w, h = _size(rng)
        cw, ch = _cell(rng, 30, 60)
        return dict(kind=kind, w=w, h=h, targets=rng.randint(1, 3), cw=cw, ch=ch,
                    levels=_levels(rng, w, h), iters=rng.choice([3, 5, 5]))
    n = _log(rng, 64, 1024)
    return dict(kind="train", n=n, pool=n * rng.randint(2, 8), radius=rng.choice([1.0, 3.0]))


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _texture(g, size):
    """Band-limited noise, periodic: uniform noise, Gaussian of 2 px."""
    t = torch.rand((size, size), generator=g, device=DEV)
    taps = [math.exp(-0.5 * (i / 2.0) ** 2) for i in range(-8, 9)]
    for d in (0, 1):
        acc = torch.zeros_like(t)
        for i, a in zip(range(-8, 9), taps):
            acc += a * torch.roll(t, i, d)
        t = acc
    return 128.0 + 40.0 * (t - t.mean()) / t.std()


def _render(tex, pose, w, h, g, disparity=0.0):
    """uint8 image (h, w) of the texture under pose (scale, angle, tx, ty); the
    camera sits `disparity` * (5 + 25 y / h) px to the right."""
    s, th, tx, ty = pose
    size = tex.shape[0]
    ys, xs = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float32),
                            torch.arange(w, device=DEV, dtype=torch.float32), indexing="ij")
    if disparity:
        xs = xs + disparity * (5.0 + 25.0 * ys / h)
    c, sn = s * math.cos(th), s * math.sin(th)
    xs, ys = xs - (w - 1) / 2, ys - (h - 1) / 2
    grid = torch.stack([c * xs - sn * ys + tx, sn * xs + c * ys + ty], -1) * (2.0 / (size - 1))
    v = nnf.grid_sample(tex[None, None], grid[None], mode="bicubic", padding_mode="reflection",
                        align_corners=True)[0, 0]
    v = v + 2.0 * torch.randn((h, w), generator=g, device=DEV)
    return torch.floor(v + 0.5).clamp_(0, 255).to(torch.uint8)


def _tex_size(w):
    return 4096 if w > 1000 else 2048


def _poses(rng, n, motion):
    """A smooth camera path: at most `motion` px a frame."""
    a, v = rng.uniform(0, 2 * math.pi), motion * rng.uniform(0.4, 0.8)
    x, y, th, s = rng.uniform(-50, 50), rng.uniform(-50, 50), rng.uniform(-0.1, 0.1), 1.0
    dth, ds = rng.uniform(-1, 1) * 1e-4 * motion, rng.uniform(-1, 1) * 5e-5 * motion
    out = []
    for _ in range(n):
        out.append((s, th, x, y))
        a += rng.uniform(-0.2, 0.2)
        x, y, th, s = x + v * math.cos(a), y + v * math.sin(a), th + dth, s * (1 + ds)
    return out


def _stereo_loop(seed, stream, w, h, steps, motion):
    """(steps, 2, h, w): a path played forward and back, a closed loop."""
    g = _gen(seed * 64 + stream)
    rng = np.random.default_rng(seed * 64 + stream)
    tex = _texture(g, _tex_size(w))
    m = steps // 2
    imgs = [torch.stack([_render(tex, p, w, h, g), _render(tex, p, w, h, g, 1.0)])
            for p in _poses(rng, m + 1, motion)]
    order = list(range(m + 1)) + list(range(m - 1, 0, -1))
    return torch.stack([imgs[i] for i in order])


def _sequence(seed, w, h, n, motion):
    """(n, h, w): consecutive frames of one camera."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    tex = _texture(g, _tex_size(w))
    return torch.stack([_render(tex, p, w, h, g) for p in _poses(rng, n, motion)])


def _corners(imgs, cw, ch, border=9):
    """(n, cells, 2) integer positions: each full cell's pixel with the largest
    minimum eigenvalue of the structure tensor, away from the border."""
    n, h, w = imgs.shape
    gx, gy = w // cw, h // ch
    out = []
    for im in imgs:
        f = im.float()
        dx = torch.zeros_like(f)
        dy = torch.zeros_like(f)
        dx[:, 1:-1] = f[:, 2:] - f[:, :-2]
        dy[1:-1] = f[2:] - f[:-2]
        a, b, c = (nnf.avg_pool2d(v[None, None], 5, 1, 2)[0, 0] for v in (dx * dx, dx * dy, dy * dy))
        e = 0.5 * (a + c) - torch.sqrt(0.25 * (a - c) ** 2 + b * b)
        e[:border] = -1
        e[h - border:] = -1
        e[:, :border] = -1
        e[:, w - border:] = -1
        cells = e[: gy * ch, : gx * cw].reshape(gy, ch, gx, cw).permute(0, 2, 1, 3)
        i = cells.reshape(gy * gx, ch * cw).argmax(1)
        cy = torch.arange(gy * gx, device=DEV) // gx * ch + i // cw
        cx = torch.arange(gy * gx, device=DEV) % gx * cw + i % cw
        out.append(torch.stack([cx, cy], -1).float())
    return torch.stack(out)


def _track_inputs(case, seed):
    """Frames and sub-pixel keypoints of every frame but the last; a prior
    start (as a motion model gives it) when tracking starts below the top."""
    imgs = _sequence(seed, case["w"], case["h"], case["pairs"] + 1, case["motion"])
    g = _gen(seed + 1)
    pts = _corners(imgs[:-1], case["cw"], case["ch"])
    pts = pts + torch.rand(pts.shape, generator=g, device=DEV) - 0.5
    init = None
    if case.get("start", -1) >= 0:
        rng = np.random.default_rng(seed)
        w, h = case["w"], case["h"]
        pose = _poses(rng, case["pairs"] + 1, case["motion"])
        flow = []
        for (s0, t0, x0, y0), (s1, t1, x1, y1) in zip(pose[:-1], pose[1:]):
            p = pts[len(flow)] - torch.tensor([(w - 1) / 2, (h - 1) / 2], device=DEV)
            c, s = s0 * math.cos(t0), s0 * math.sin(t0)
            X, Y = c * p[:, 0] - s * p[:, 1] + x0 - x1, s * p[:, 0] + c * p[:, 1] + y0 - y1
            c, s = math.cos(t1) / s1, math.sin(t1) / s1
            flow.append(torch.stack([c * X + s * Y + (w - 1) / 2, -s * X + c * Y + (h - 1) / 2,
                                     torch.full_like(X, t0 - t1)], -1))
        init = torch.stack(flow)
        init[..., :2] += torch.randn(init[..., :2].shape, generator=g, device=DEV) * 0.7
        init = init.contiguous()
    return imgs, pts.contiguous(), init


def _rig_inputs(case, seed):
    """A source image, its keypoints and inverse depths (2% off), targets at
    growing baselines, and their poses."""
    w, h, nt = case["w"], case["h"], case["targets"]
    g, rng = _gen(seed), np.random.default_rng(seed)
    tex = _texture(g, _tex_size(w))
    pose = _poses(rng, 1, 1.0)[0]
    base = [0.6 + 0.5 * j for j in range(nt)]
    imgs = torch.stack([_render(tex, pose, w, h, g, b) for b in [0.0] + base])
    pts = _corners(imgs[:1], case["cw"], case["ch"])
    rho = (5.0 + 25.0 * pts[..., 1] / h) / 500.0
    rho = rho * (1 + 0.02 * torch.randn(rho.shape, generator=g, device=DEV))
    poses = torch.zeros((nt, 12), device=DEV)
    poses[:, 0] = poses[:, 4] = poses[:, 8] = 1.0
    poses[:, 9] = -torch.tensor(base, device=DEV)
    poses[:, 11] = 0.001
    K = (500.0, 500.0, (w - 1) / 2, (h - 1) / 2)
    return imgs, pts.repeat(nt, 1, 1).contiguous(), rho.repeat(nt, 1).contiguous(), poses, K


def _train_inputs(case, seed):
    """A pool of network inputs (source and target patches at two levels, byte
    values as BF16) with their flows, and one minibatch's indices."""
    g, n = _gen(seed), case["pool"]
    tex = _texture(g, 1024)
    flow = (torch.rand((n, 2), generator=g, device=DEV) * 2 - 1) * 40.0
    c = torch.rand((n, 2), generator=g, device=DEV) * 900.0
    r = torch.arange(16, device=DEV) - 8
    xs = []
    for lv in (2, 3):
        d = 4.0 if lv == 2 else 8.0
        for off in (torch.zeros_like(flow), flow):
            x = torch.floor((c[:, 0] + off[:, 0]) / d * 2 + 0.5).long()[:, None, None] + 2 * r
            y = torch.floor((c[:, 1] + off[:, 1]) / d * 2 + 0.5).long()[:, None, None] + 2 * r[:, None]
            xs.append(tex[y % 1024, x % 1024])
    v = torch.stack(xs, 1)
    v = v + 1.5 * torch.randn(v.shape, generator=g, device=DEV)
    x = (torch.floor(v + 0.5).clamp(0, 255) - 128.0) / 64.0
    x = x.to(torch.bfloat16).view(torch.int16).contiguous()
    index = torch.randperm(n, generator=g, device=DEV)[: case["n"]].to(torch.int32)
    return x, flow.contiguous(), index.contiguous()


# ----------------------------------------------------------------- prepare --
def _params(case, **kw):
    t = [v for v in (40, 20, 10, 5) if v >= case.get("tmin", 5)]
    return vio.default_params(n_levels=case["levels"], gn_iters=case.get("iters", 5),
                              cell_w=case.get("cw", 50), cell_h=case.get("ch", 50),
                              k_per_cell=case.get("k", 1), thresholds=t, **kw)


def _f(*shape):
    return torch.zeros(shape, dtype=torch.float32, device=DEV)


def _u8(*shape):
    return torch.zeros(shape, dtype=torch.uint8, device=DEV)


def _levels_of(pyr):
    """The upper levels of every image, (n, h, w) each."""
    L, n, ub = pyr.layout, pyr.n, int(pyr.layout.upper_bytes)
    return [torch.as_strided(pyr.upper, (n, L.h[l], L.w[l]), (ub, L.pitch[l], 1), int(L.offset[l]))
            for l in range(1, L.n_levels)]


def _pyramids(imgs, levels):
    pyr = vio.Pyramids(imgs, levels)
    pyr.upper.zero_()
    return pyr


def _owned(view, owner):
    """The tensors of a view, each keeping the object whose memory it shows."""
    view = {k: v for k, v in view.items() if k != "parity"}
    for v in view.values():
        v.owner = owner
    return view


def prepare(case, seed):
    kind = case["kind"]
    if kind == "frame":
        w, h, ns = case["w"], case["h"], case["streams"]
        frames = torch.stack([_stereo_loop(seed, s, w, h, case["steps"], case["motion"])
                              for s in range(ns)], 1).contiguous()
        cap = 2 * (w // case["cw"]) * (h // case["ch"]) * case["k"]
        fe = vio.Frontend(_params(case), w, h, ns, cap)
        st = dict(case=case, fe=fe, frames=frames, steps=list(frames))
        if case["learned"]:
            st["net"] = vio.InitNet.load(WEIGHTS)
            fe.set_initnet(st["net"])
        torch.cuda.synchronize()
        fe.run(frames)          # a session in progress
        torch.cuda.synchronize()
        # the step count is even: the same buffers after every pass
        st["view"] = _owned(fe.view(), fe)
        return st
    if kind == "batch":
        groups, loops = [], []
        for gi, spec in enumerate(case["groups"].split()):
            size, cell = spec.split("/")
            w, h, ns = (int(v) for v in size.split("x"))
            cw, ch = (int(v) for v in cell.split("x"))
            p = vio.default_params(n_levels=case["levels"], cell_w=cw, cell_h=ch)
            groups.append((p, w, h, ns, 2 * (w // cw) * (h // ch)))
            loops.append([_stereo_loop(seed, 8 * gi + s, w, h, 2, case["motion"])
                          for s in range(ns)])
        b = vio.Batch(groups)
        st = dict(case=case, batch=b, stream=torch.cuda.Stream())
        if case["learned"]:
            st["net"] = vio.InitNet.load(WEIGHTS)
            b.set_initnet(st["net"])
        b.set_graph(case["graph"])
        torch.cuda.synchronize()
        with torch.cuda.stream(st["stream"]):
            for t in range(2):   # both frame slots of every stream, tracks on the device
                for gi, g in enumerate(loops):
                    for s, fr in enumerate(g):
                        b.next_frame(gi, s).copy_(fr[t])
                b.step()
        torch.cuda.synchronize()
        st["out"] = [_owned(b.view(gi), b) for gi in range(len(groups))]
        return st
    if kind == "detect":
        w, h, n = case["w"], case["h"], case["n"]
        g, rng = _gen(seed), np.random.default_rng(seed)
        tex = _texture(g, _tex_size(w))
        imgs = torch.stack([_render(tex, (rng.uniform(0.9, 1.1), rng.uniform(-0.5, 0.5),
                                          rng.uniform(-300, 300), rng.uniform(-300, 300)), w, h, g)
                            for _ in range(n)])
        cells = (w // case["cw"]) * (h // case["ch"])
        cap = max(1, cells * case["k"])
        st = dict(case=case, pyr=_pyramids(imgs, case["levels"]), cap=cap, kp=_f(n, cap, 2),
                  score=torch.zeros((n, cap), dtype=torch.int16, device=DEV),
                  count=torch.zeros(n, dtype=torch.int32, device=DEV), opt={},
                  ctx=vio.Context(_params(case, round_mode=case["rnd"],
                                          select_mode=case["select"]), w, h, n))
        if case["mask"]:        # a dark disc at the bottom of the image and a strip
            ys, xs = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV),
                                    indexing="ij")
            m = ((xs - w // 2) ** 2 + (ys - h) ** 2 > (h // 3) ** 2) & (xs > w // 20)
            st["opt"].update(mask=m.to(torch.uint8).repeat(n, 1, 1).contiguous(), mask_stride=w * h)
        if case["occ"]:
            o = torch.rand((n, max(cells, 1)), generator=g, device=DEV)
            st["opt"]["occupancy"] = (o * (case["k"] + 1)).to(torch.uint8)
        st["levels"] = _levels_of(st["pyr"])
        st["b"] = st["pyr"].batch()
        return st
    if kind in ("track", "propose"):
        imgs, pts, init = _track_inputs(case, seed)
        n, cap = pts.shape[:2]
        pyr = _pyramids(imgs, case["levels"])
        ctx = vio.Context(_params(case), case["w"], case["h"], n + 1)
        ctx.pyramid_build(pyr)
        st = dict(case=case, pyr=pyr, ctx=ctx, src=pyr.batch(0, 1, n), dst=pyr.batch(1, 1, n),
                  pts=pts, cap=cap, count=torch.full((n,), cap, dtype=torch.int32, device=DEV))
        if kind == "propose":
            st.update(net=vio.InitNet.load(WEIGHTS), out=_f(n * cap, 3),
                      x=torch.zeros((n * cap, 4, 16, 16), dtype=torch.int16, device=DEV))
        else:
            st.update(init=init, out=_f(n, cap, 3), status=_u8(n, cap), fb=_f(n, cap),
                      last=_f(n, cap))
        return st
    if kind == "rig":
        imgs, pts, rho, poses, K = _rig_inputs(case, seed)
        nt, cap = rho.shape
        pyr = _pyramids(imgs, case["levels"])
        ctx = vio.Context(_params(case), case["w"], case["h"], nt + 1)
        ctx.pyramid_build(pyr)
        return dict(case=case, pyr=pyr, ctx=ctx, src=pyr.batch(0, 1, 1), dst=pyr.batch(1, 1, nt),
                    pts=pts, one=pts[0].contiguous(), rho=rho, poses=poses, K=K, cap=cap, nt=nt,
                    init=_f(nt, cap, 3), valid=_u8(nt, cap), match=_f(nt, cap, 2),
                    status=_u8(nt, cap), fb=_f(nt, cap))
    x, flow, index = _train_inputs(case, seed)
    net = vio.InitNet.load(WEIGHTS)      # resumes from the shipped moments and step
    return dict(case=case, net=net, x=x, flow=flow, index=index,
                grad=torch.zeros_like(net.master), loss=_f(1))


# --------------------------------------------------------------------- run --
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "frame":
        if case["piped"]:
            st["fe"].run(st["frames"])
        else:
            for f in st["steps"]:
                st["fe"].step(f)
        return st["view"]
    if kind == "batch":
        st["batch"].step(stream=st["stream"])
        return st["out"]
    if kind == "detect":
        if case["fused"]:
            st["ctx"].pyramid_detect(st["pyr"], st["kp"], st["score"], st["count"], st["cap"],
                                     **st["opt"])
        else:
            st["ctx"].pyramid_build(st["pyr"])
            st["ctx"].detect_grid(st["pyr"], st["b"], st["kp"], st["score"], st["count"],
                                  st["cap"], **st["opt"])
        return dict(kp=st["kp"], score=st["score"], count=st["count"], levels=st["levels"])
    if kind == "track":
        st["ctx"].track_patches(st["pyr"], st["src"], st["dst"], st["pts"], st["count"], st["cap"],
                                st["out"], st["status"], st["fb"], init=st["init"],
                                fb=case["fb"], last_step=st["last"],
                                from_level=case["start"] if case["start"] >= 0 else None)
        return dict(out=st["out"], status=st["status"], fb=st["fb"], last=st["last"])
    if kind == "rig":
        vio.predict_warp(st["K"], st["K"], st["poses"], st["pts"], st["rho"], None, st["cap"],
                         st["nt"], st["init"], st["valid"])
        st["ctx"].match_cameras(st["pyr"], st["src"], st["dst"], st["one"], None, st["cap"],
                                st["match"], st["status"], st["fb"], init=st["init"])
        return dict(init=st["init"], valid=st["valid"], match=st["match"], status=st["status"],
                    fb=st["fb"])
    if kind == "propose":
        vio.initnet_extract(st["pyr"], st["src"], st["dst"], st["pts"], st["count"], st["cap"],
                            case["la"], case["lb"], st["x"])
        st["net"].forward(st["x"], st["out"])
        return dict(x=st["x"], out=st["out"])
    net, n = st["net"], case["n"]
    net.pack()
    st["grad"].zero_()
    st["loss"].zero_()
    vio.initnet_train_step(net.packed, st["x"], st["flow"], st["index"], n, 1.0 / n, st["grad"],
                           st["loss"], label_radius=case["radius"])
    net.step += 1
    vio.initnet_adam(net.master, st["grad"], net.m, net.v, net.step, 1e-4)
    return dict(grad=st["grad"], loss=st["loss"], master=net.master, m=net.m, v=net.v)


# -------------------------------------------------------------------- work --
def _upper(w, h, levels):
    return sum((w >> l) * (h >> l) for l in range(1, levels))


_FAST_OPS = 60        # a FAST score: 16 differences and the arc minima and maxima
_NET_FLOPS = 2 * (64 * 32 * 36 + 16 * 32 * 288 + 4 * 32 * 288 + 128 * 64 + 64 * 3)


def _track_flops(levels, iters, directions):
    return directions * levels * (52 * 72 + iters * 52 * 26)


def _image_work(w, h, levels, cells, k):
    """Level 0 read, upper levels written, the keypoints written."""
    return w * h + _upper(w, h, levels) + 10 * cells * k, 5 * _upper(w, h, levels) * 2 + _FAST_OPS * w * h


def work(case):
    kind = case["kind"]
    if kind in ("frame", "batch"):
        if kind == "frame":
            groups = [(case["w"], case["h"], case["streams"], case["cw"], case["ch"], case["k"])]
            steps, iters = case["steps"], case["iters"]
        else:
            groups, steps, iters = [], 1, 5
            for spec in case["groups"].split():
                size, cell = spec.split("/")
                groups.append(tuple(int(v) for v in (size + "x" + cell).split("x")) + (1,))
        nbytes = flops = 0
        for w, h, ns, cw, ch, k in groups:
            cells = (w // cw) * (h // ch)
            b, f = _image_work(w, h, case["levels"], cells, k)
            # both cameras' pyramids, the previous levels read for tracking, lists
            nbytes += ns * (2 * (2 * w * h + _upper(w, h, case["levels"])) + 4 * cells * k * 13)
            # detection on one camera; two cameras' tracks, forward and backward
            flops += ns * (f + 2 * cells * k * _track_flops(case["levels"], iters, 2))
            if case["learned"]:
                flops += ns * 2 * cells * k * _NET_FLOPS
        return {"bytes": float(steps * nbytes), "flops": float(steps * flops)}
    if kind == "train":
        n = case["n"]
        return {"bytes": float(n * (2048 + 8 + 4) + 28131 * 4 * 8), "flops": float(3 * n * _NET_FLOPS)}
    cells = (case["w"] // case["cw"]) * (case["h"] // case["ch"])
    if kind == "detect":
        b, f = _image_work(case["w"], case["h"], case["levels"], cells, case["k"])
        return {"bytes": float(case["n"] * (b + (case["w"] * case["h"] if case["mask"] else 0))),
                "flops": float(case["n"] * f)}
    if kind == "rig":
        n, per_image, images = cells * case["targets"], cells, case["targets"] + 1
        pix = case["w"] * case["h"] + _upper(case["w"], case["h"], case["levels"])
        return {"bytes": float(min(images * pix, 2 * n * case["levels"] * 324) + n * 41 + per_image * 8),
                "flops": float(n * (53 * 30 + _track_flops(case["levels"], case["iters"], 2)))}
    n = case["pairs"] * cells
    pix = (case["pairs"] + 1) * (case["w"] * case["h"] + _upper(case["w"], case["h"], case["levels"]))
    if kind == "propose":
        return {"bytes": float(min(pix, n * 4 * 256) + n * (8 + 2048 + 12)),
                "flops": float(n * _NET_FLOPS)}
    levels = case["levels"] if case["start"] < 0 else case["start"] + 1
    return {"bytes": float(min(pix, 2 * n * levels * 324) + n * (8 + 21)),
            "flops": float(n * _track_flops(levels, case["iters"], 2 if case["fb"] else 1))}


# ------------------------------------------------------------------- exact --
def _pyramid64(imgs, levels):
    """Integer pyramid: 5x5 binomial, edges clamped, rounded to nearest."""
    out, cur = [imgs.to(torch.float64)], imgs.to(torch.int64)
    k = (1, 4, 6, 4, 1)
    for _ in range(1, levels):
        n, h, w = cur.shape
        ys = [(2 * torch.arange(h // 2, device=DEV) + i - 2).clamp(0, h - 1) for i in range(5)]
        xs = [(2 * torch.arange(w // 2, device=DEV) + i - 2).clamp(0, w - 1) for i in range(5)]
        v = sum(k[i] * cur[:, ys[i]] for i in range(5))
        cur = (sum(k[i] * v[:, :, xs[i]] for i in range(5)) + 128) >> 8
        out.append(cur.to(torch.float64))
    return out


def _pattern():
    p = [(u, v) for v in range(-7, 8, 2) for u in range(-7, 8, 2) if abs(u) + abs(v) <= 10]
    return torch.tensor(p, dtype=torch.float64, device=DEV).unbind(1)


def _sample(im, idx, x, y):
    """Bilinear samples of image idx (per keypoint) at (x, y), clamped reads."""
    n, h, w = im.shape
    fx, fy = torch.floor(x), torch.floor(y)
    ix, iy = fx.long().clamp(0, w - 2), fy.long().clamp(0, h - 2)
    flat, o = im.reshape(-1), idx[:, None] * (h * w) + iy * w + ix
    ax, ay = x - fx, y - fy
    top = flat[o] * (1 - ax) + flat[o + 1] * ax
    bot = flat[o + w] * (1 - ax) + flat[o + w + 1] * ax
    return top * (1 - ay) + bot * ay


def _track64(src, si, dst, di, p, t, th, iters, top):
    """Inverse-compositional tracking in 64 bits: (t, theta, ok, last step)."""
    U, V = _pattern()
    t, th = t / 2.0 ** top, th.clone()
    ok = torch.ones(len(p), dtype=torch.bool, device=DEV)
    last = torch.zeros(len(p), dtype=torch.float64, device=DEV)
    for l in range(top, -1, -1):
        S, D = src[l], dst[l]
        q = p / 2.0 ** l
        cx, cy = q[:, :1] + U, q[:, 1:] + V
        sh, sw = S.shape[1:]
        good = ((cx >= 1) & (cx < sw - 2) & (cy >= 1) & (cy < sh - 2)).all(1)
        s = _sample(S, si, cx, cy)
        gx = 0.5 * (_sample(S, si, cx + 1, cy) - _sample(S, si, cx - 1, cy))
        gy = 0.5 * (_sample(S, si, cx, cy + 1) - _sample(S, si, cx, cy - 1))
        mean = s.mean(1, keepdim=True)
        J = torch.stack([gx, gy, gy * U - gx * V], -1) / mean[..., None]
        H = J.transpose(1, 2) @ J
        good &= mean[:, 0] > 0
        tr = H.diagonal(dim1=1, dim2=2).sum(1)
        C, bad = torch.linalg.cholesky_ex(torch.where(good[:, None, None], H,
                                                      torch.eye(3, device=DEV, dtype=H.dtype)))
        good &= (bad == 0) & ((C.diagonal(dim1=1, dim2=2) ** 2).min(1).values > 1e-9 * tr)
        C = torch.where(good[:, None, None], C, torch.eye(3, device=DEV, dtype=H.dtype))
        if l == 0:
            ok &= good
        for it in range(iters):
            c, sn = torch.cos(th)[:, None], torch.sin(th)[:, None]
            x, y = c * U - sn * V + t[:, :1], sn * U + c * V + t[:, 1:]
            dh, dw = D.shape[1:]
            step = ok & good
            inside = ((x >= 0) & (x < dw - 1) & (y >= 0) & (y < dh - 1)).all(1)
            r = _sample(D, di, x.nan_to_num(0, 0, 0).clamp(-1e6, 1e6),
                        y.nan_to_num(0, 0, 0).clamp(-1e6, 1e6))
            rm = r.mean(1, keepdim=True)
            e = r / rm - s / mean
            d = -torch.cholesky_solve((J * e[..., None]).sum(1)[..., None], C)[..., 0]
            fine = inside & (rm[:, 0] > 0) & torch.isfinite(d).all(1)
            ok &= ~step | fine
            step &= fine
            a = torch.where(d[:, 2].abs() < 1e-9, 1 - d[:, 2] ** 2 / 6, torch.sin(d[:, 2]) / d[:, 2])
            b = torch.where(d[:, 2].abs() < 1e-9, 0.5 * d[:, 2], (1 - torch.cos(d[:, 2])) / d[:, 2])
            vx, vy = a * d[:, 0] - b * d[:, 1], b * d[:, 0] + a * d[:, 1]
            c, sn = c[:, 0], sn[:, 0]
            new = torch.stack([t[:, 0] + c * vx - sn * vy, t[:, 1] + sn * vx + c * vy], -1)
            t = torch.where(step[:, None], new, t)
            th = torch.where(step, th + d[:, 2], th)
            if l == 0 and it == iters - 1:
                last = d[:, 0].abs() + d[:, 1].abs() + math.hypot(7, 3) * d[:, 2].abs()
        if l > 0:
            t = t * 2
    return t, th, ok, last


def _track_fb64(levels, si, di, p, t0, th0, iters, top, fb):
    t, th, ok, last = _track64(levels, si, levels, di, p, t0, th0, iters, top)
    nan = torch.full_like(last, float("nan"))
    dist = nan
    if fb:
        tb, _, okb, _ = _track64(levels, di, levels, si, torch.where(ok[:, None], t, p), p, -th,
                                 iters, top)
        dist = torch.where(ok & okb, torch.linalg.norm(tb - p, dim=1), nan)
    out = torch.where(ok[:, None], torch.cat([t, th[:, None]], 1), nan[:, None])
    return out, dist, torch.where(ok, last, nan)


def _weights64():
    """The network's weights as inference uses them (BF16 values), biases, and
    the master vector, in 64 bits."""
    with np.load(WEIGHTS, allow_pickle=False) as z:
        m = torch.from_numpy(z["master"]).to(DEV)
        mom = [torch.from_numpy(z[k]).to(DEV).double() for k in ("m", "v")]
        step = int(z["step"][0])
    shapes = [(32, 4, 3, 3), (32,), (32, 32, 3, 3), (32,), (32, 32, 3, 3), (32,), (64, 128), (64,),
              (3, 64), (3,)]
    parts, at = [], 0
    for s in shapes:
        n = int(np.prod(s))
        v = m[at:at + n].reshape(s)
        parts.append((v.to(torch.bfloat16) if len(s) > 1 else v).double().requires_grad_())
        at += n
    return parts, m.double(), mom, step


def _net64(P, x):
    for i in (0, 2, 4):
        x = torch.relu(nnf.conv2d(x, P[i], P[i + 1], stride=2, padding=1))
    x = torch.relu(x.flatten(1) @ P[6].t() + P[7])
    return x @ P[8].t() + P[9]


def exact(case, seed):
    """Tracked positions, predicted starts, proposals and training steps in 64
    bits. A session's lists and the detections are whole-number decisions (or
    follow from them): no value."""
    kind = case["kind"]
    if kind in ("frame", "batch", "detect"):
        return None
    if kind == "rig":
        imgs, pts, rho, poses, (f, _, cx, cy) = _rig_inputs(case, seed)
        nt, cap = rho.shape
        U, V = _pattern()
        p, z, T = pts.double(), 1 / rho.double(), poses.double()

        def project(x, y, z):
            X, Y = (x - cx) * z / f, (y - cy) * z / f
            q = [T[:, 3 * i, None, None] * X + T[:, 3 * i + 1, None, None] * Y
                 + T[:, 3 * i + 2, None, None] * z + T[:, 9 + i, None, None] for i in range(3)]
            return f * q[0] / q[2] + cx, f * q[1] / q[2] + cy
        tx, ty = project(p[..., :1], p[..., 1:], z[..., None])
        yx, yy = project(p[..., :1] + U, p[..., 1:] + V, z[..., None])
        th = torch.atan2((U * (yy - ty) - V * (yx - tx)).sum(-1), (U * (yx - tx) + V * (yy - ty)).sum(-1))
        init = torch.cat([tx, ty, th[..., None]], -1)
        L = _pyramid64(imgs, case["levels"])
        di = 1 + torch.arange(nt * cap, device=DEV) // cap
        out, dist, _ = _track_fb64(L, torch.zeros_like(di), di, p.reshape(-1, 2),
                                   init[..., :2].reshape(-1, 2), th.reshape(-1), case["iters"],
                                   case["levels"] - 1, True)
        return dict(init=init, valid=None, match=out[:, :2].reshape(nt, cap, 2), status=None,
                    fb=dist.reshape(nt, cap))
    if kind == "track":
        imgs, pts, init = _track_inputs(case, seed)
        n, cap = pts.shape[:2]
        top = case["start"] if case["start"] >= 0 else case["levels"] - 1
        p = pts.double().reshape(-1, 2)
        t0 = init.double().reshape(-1, 3) if init is not None else torch.cat([p, 0 * p[:, :1]], 1)
        si = torch.arange(n * cap, device=DEV) // cap
        out, dist, last = _track_fb64(_pyramid64(imgs, case["levels"]), si, si + 1, p, t0[:, :2],
                                      t0[:, 2], case["iters"], top, case["fb"])
        return dict(out=out.reshape(n, cap, 3), status=None, fb=dist.reshape(n, cap),
                    last=last.reshape(n, cap))
    P, master, (m, v), step = _weights64()
    if kind == "propose":
        imgs, pts, _ = _track_inputs(case, seed)
        n, cap = pts.shape[:2]
        L = _pyramid64(imgs, case["levels"])
        r = torch.arange(16, device=DEV) - 8
        img = torch.arange(n, device=DEV)[:, None, None, None]
        chans = []
        for l in (case["la"], case["lb"]):
            c = torch.floor(pts.double() / 2 ** l + 0.5).long()
            x, y = c[..., 0, None, None] + r, c[..., 1, None, None] + r[:, None]
            h, w = L[l].shape[1:]
            inside = (x >= 0) & (x < w) & (y >= 0) & (y < h)
            for k in (0, 1):
                val = L[l][img + k, y.clamp(0, h - 1), x.clamp(0, w - 1)]
                chans.append(torch.where(inside, (val - 128) / 64, torch.zeros_like(val)))
        x = torch.stack(chans, 2).reshape(n * cap, 4, 16, 16)
        with torch.no_grad():
            o = torch.cat([_net64(P, x[i:i + 4096]) for i in range(0, len(x), 4096)])
        return dict(x=None, out=torch.cat([16.0 * o[:, :2], torch.sigmoid(o[:, 2:])], 1))
    x, flow, index = _train_inputs(case, seed)
    i = index.long()
    x, f = x.view(torch.bfloat16)[i].double(), flow[i].double()
    o = _net64(P, x)
    y = (torch.linalg.norm(16.0 * o[:, :2] - f, dim=1) < case["radius"]).double()
    loss = ((o[:, :2] - f / 16.0) ** 2).sum() + nnf.binary_cross_entropy_with_logits(
        o[:, 2], y.detach(), reduction="sum")
    loss.backward()
    g = torch.cat([q.grad.reshape(-1) for q in P]) / len(x)
    t = step + 1
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    master = master - 1e-4 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return dict(grad=g, loss=loss.detach().reshape(1), master=master, m=m, v=v)
