"""Launches large enough for the grouped tracker against the same keypoints in
launches that keep a warp each, bit for bit: the stage call with starts,
counts, start levels and rows at any byte, and frame steps with and without
the learned start."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")
from test_gpu_front_split import _frames  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)


@pytest.mark.parametrize("w,h,levels,fb,init,start", [
    (320, 240, 4, True, False, None),     # rows on 16-byte boundaries
    (331, 203, 3, True, True, 1),         # level 0 at any byte
    (300, 211, 2, False, True, None),     # level 0 on words
])
def test_stage_call(w, h, levels, fb, init, start):
    lim = 28 * torch.cuda.get_device_properties(0).multi_processor_count
    frames = _frames(w, h, 2, w)[:, 0].contiguous()
    pyr = vio.Pyramids(frames, levels)
    ctx = vio.Context(vio.default_params(n_levels=levels), w, h, 2)
    ctx.pyramid_build(pyr)
    cap = lim + 77
    g = torch.Generator().manual_seed(w)
    pts = torch.rand((1, cap, 2), generator=g) * torch.tensor([w + 20.0, h + 20.0]) - 10.0
    ini = torch.cat([pts + torch.randn((1, cap, 2), generator=g) * 3,
                     0.1 * torch.randn((1, cap, 1), generator=g)], 2)
    ini[0, 5, 0], ini[0, 6, 1], pts[0, 7, 0] = 1e30, float("nan"), float("nan")
    pts, ini = pts.cuda(), ini.cuda().contiguous() if init else None
    count = torch.tensor([cap - 13], dtype=torch.int32, device="cuda")

    def call(lo, hi, n):
        m = hi - lo
        out = torch.zeros((1, m, 3), device="cuda")
        st = torch.zeros((1, m), dtype=torch.uint8, device="cuda")
        d, last = torch.zeros((1, m), device="cuda"), torch.zeros((1, m), device="cuda")
        ctx.track_patches(pyr, pyr.batch(0, 1, 1), pyr.batch(1, 1, 1), pts[:, lo:hi].contiguous(), n,
                          m, out, st, d, init=ini[:, lo:hi].contiguous() if init else None, fb=fb,
                          from_level=start, last_step=last)
        return [t.view(torch.int32) if t.dtype == torch.float32 else t for t in (out, st, d, last)]
    whole = call(0, cap, count)
    half = cap // 2
    parts = [call(0, half, None),
             call(half, cap, torch.tensor([cap - 13 - half], dtype=torch.int32, device="cuda"))]
    for i, a in enumerate(whole):
        assert torch.equal(a, torch.cat([p[i] for p in parts], 1)), i
    assert (whole[1] == 0).sum() > 1000 and (whole[1] == 255).sum() == 13


@pytest.mark.parametrize("learned", [False, True])
def test_frame_steps(learned):
    w, h, L, cell, ns = 640, 480, 4, 16, 6
    p = vio.default_params(n_levels=L, cell_w=cell, cell_h=cell)
    cells = (w // cell) * (h // cell)
    cap = 2 * cells
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert ns * (2 * cap + cells) >= 200 * sms > 2 * cap + cells
    net = None
    if learned:
        flat = torch.randn(vio.INITNET_N_PARAMS, generator=torch.Generator().manual_seed(3)) * 0.05
        net = vio.InitNet(flat, 2, 3, 1, 0.5)
    frames = [_frames(w, h, 4, 50 + s) for s in range(ns)]
    b = vio.Batch([(p, w, h, ns, cap)])
    if net is not None:
        b.set_initnet(net)
    for t in range(4):
        for s in range(ns):
            b.next_frame(0, s).copy_(frames[s][t])
        b.step()
    torch.cuda.synchronize()
    for s in range(ns):
        fe = vio.Frontend(p, w, h, 1, cap)
        if net is not None:
            fe.set_initnet(net)
        for t in range(4):
            fe.step(frames[s][t].view(1, 2, h, w))
        torch.cuda.synchronize()
        v = fe.view()
        xy, ids = b.stream_lists(0, s)
        for c in range(2):
            n = int(v["track_count"][0, c])
            assert n > 0 and np.array_equal(ids[c], v["track_id"][0, c, :n].cpu().numpy())
            assert np.array_equal(xy[c], v["track_xy"][0, c, :n].cpu().numpy())
