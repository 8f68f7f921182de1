"""The grouped tracker on level-0 rows that start at any byte, in launches large
enough for it, against launches that keep a warp per keypoint, bit for bit;
keypoints over the whole image and around its corners."""
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


@pytest.mark.parametrize("w,h,levels,init", [
    (331, 203, 3, True),
    (322, 97, 2, False),
    (65, 49, 1, True),      # most windows touch an edge
])
def test_any_byte_rows(w, h, levels, init):
    lim = 48 * torch.cuda.get_device_properties(0).multi_processor_count
    frames = _frames(w, h, 2, w)[:, 0].contiguous()
    pyr = vio.Pyramids(frames, levels)
    ctx = vio.Context(vio.default_params(n_levels=levels), w, h, 2)
    ctx.pyramid_build(pyr)
    cap = lim + 41
    g = torch.Generator().manual_seed(w)
    size = torch.tensor([float(w), float(h)])
    pts = torch.rand((1, cap, 2), generator=g) * size
    corner = (torch.rand((1, 800, 2), generator=g) < 0.5).float() * (size - 24.0)
    pts[:, :800] = corner + torch.rand((1, 800, 2), generator=g) * 24.0
    pts = pts.cuda()
    ini = None
    if init:
        ini = torch.cat([pts.cpu() + torch.randn((1, cap, 2), generator=g) * 2,
                         0.05 * torch.randn((1, cap, 1), generator=g)], 2).cuda().contiguous()

    def call(lo, hi):
        m = hi - lo
        out = torch.zeros((1, m, 3), device="cuda")
        st = torch.zeros((1, m), dtype=torch.uint8, device="cuda")
        d, last = torch.zeros((1, m), device="cuda"), torch.zeros((1, m), device="cuda")
        ctx.track_patches(pyr, pyr.batch(0, 1, 1), pyr.batch(1, 1, 1), pts[:, lo:hi].contiguous(),
                          None, m, out, st, d, init=ini[:, lo:hi].contiguous() if init else None,
                          fb=True, last_step=last)
        return [t.view(torch.int32) if t.dtype == torch.float32 else t for t in (out, st, d, last)]
    whole = call(0, cap)
    parts = [call(0, cap // 2), call(cap // 2, cap)]
    for i, a in enumerate(whole):
        assert torch.equal(a, torch.cat([p[i] for p in parts], 1)), i
    assert (whole[1] == 0).sum() > 100
