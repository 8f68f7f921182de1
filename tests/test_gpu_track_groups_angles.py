"""Starts with a non-finite angle in a launch large enough for the grouped
tracker against the same keypoints in launches that keep a warp each, bit for
bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")
from test_gpu_front_split import _frames  # noqa: E402


@pytest.mark.parametrize("w,h,levels,fb", [(320, 240, 4, True), (331, 203, 1, False)])
def test_non_finite_start_angles(w, h, levels, fb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)
    lim = 48 * torch.cuda.get_device_properties(0).multi_processor_count
    pyr = vio.Pyramids(_frames(w, h, 2, w)[:, 0].contiguous(), levels)
    ctx = vio.Context(vio.default_params(n_levels=levels), w, h, 2)
    ctx.pyramid_build(pyr)
    cap = lim + 30
    g = torch.Generator().manual_seed(w)
    pts = torch.rand((1, cap, 2), generator=g) * torch.tensor([w - 40.0, h - 40.0]) + 20.0
    ini = torch.cat([pts, 0.1 * torch.randn((1, cap, 1), generator=g)], 2)
    for i, bad in enumerate((float("nan"), float("inf"), -float("inf"))):
        ini[0, i::7, 2] = bad
    pts, ini = pts.cuda(), ini.cuda()

    def call(lo, hi):
        m = hi - lo
        out = torch.zeros((1, m, 3), device="cuda")
        st = torch.zeros((1, m), dtype=torch.uint8, device="cuda")
        ctx.track_patches(pyr, pyr.batch(0, 1, 1), pyr.batch(1, 1, 1), pts[:, lo:hi].contiguous(),
                          None, m, out, st, init=ini[:, lo:hi].contiguous(), fb=fb)
        return out.view(torch.int32), st
    whole = call(0, cap)
    parts = [call(cap * i // 4, cap * (i + 1) // 4) for i in range(4)]
    for i, a in enumerate(whole):
        assert torch.equal(a, torch.cat([p[i] for p in parts], 1)), i
    assert all(int((whole[1][0, i::7] == 0).sum()) == 0 for i in range(3))
    assert int((whole[1] == 0).sum()) > 1000
