"""Network input extraction at the edges of its vector path: levels whose rows
do and do not start on word boundaries, outputs that are and are not 16-byte
aligned, keypoints over and beyond every edge, unused slots. Bit for bit
against the oracle's extraction."""
import numpy as np
import pytest
import torch

import oracle
from oracle import initnet as onet

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")


@pytest.mark.parametrize("w,h,pitch,la,lb,shift", [
    (67, 45, 67, 0, 1, 0),     # level 0 at any byte
    (64, 48, 64, 0, 2, 0),     # level 0 on words
    (97, 70, 101, 1, 2, 1),    # outputs two bytes past a 16-byte boundary
    (33, 40, 36, 1, 0, 0),
])
def test_extract_edges(w, h, pitch, la, lb, shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)
    oracle.build()
    L, rng = 3, np.random.default_rng(w)
    frames = rng.integers(0, 256, (2, h, pitch), dtype=np.uint8)
    pyr = vio.Pyramids(torch.from_numpy(frames).cuda(), L, w)
    ctx = vio.Context(vio.default_params(n_levels=L), w, h, 2)
    ctx.pyramid_build(pyr)
    pts = np.concatenate([rng.uniform(-12, [w + 12, h + 12], (40, 2)),
                          [[0, 0], [w - 1, h - 1], [-0.5, h - 0.5], [1e9, 3], [w / 2, -1e9]]])
    n, cap = len(pts), len(pts) + 3
    d_pts = torch.zeros((1, cap, 2))
    d_pts[0, :n] = torch.from_numpy(pts.astype(np.float32))
    buf = torch.full((cap * 1024 + 16,), 0x7777, dtype=torch.int16, device="cuda")
    x = buf[shift: shift + cap * 1024]
    count = torch.tensor([n], dtype=torch.int32, device="cuda")
    vio.initnet_extract(pyr, pyr.batch(0, 1, 1), pyr.batch(1, 1, 1), d_pts.cuda(), count, cap, la,
                        lb, x)
    got = x.cpu().numpy().view(np.uint16).reshape(cap, 4, 16, 16)
    lv = [[pyr.level(i, l).cpu().numpy() for l in range(L)] for i in range(2)]
    for i, (px, py) in enumerate(pts.astype(np.float32)):
        ref = onet.extract(lv[0], lv[1], float(px), float(py), la, lb)
        ref = (np.ascontiguousarray(ref, np.float32).view(np.uint32) >> 16).astype(np.uint16)
        assert np.array_equal(got[i], ref.reshape(4, 16, 16)), i
    assert not got[n:].any()
    rest = buf.cpu().numpy()
    assert (rest[:shift] == 0x7777).all() and (rest[shift + cap * 1024:] == 0x7777).all()
