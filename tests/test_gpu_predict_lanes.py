"""The model-based start of a launch small enough for eight lanes per keypoint
against the same keypoints in one launch of a thread each."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)


# Both forms project the same points. Where the compiler contracts a product
# differently, each of about ten rounded operations moves a projection by at
# most 2^-24 of its distance from the principal point (below 1100 px here), and
# the last sum by two units of 2^-13: 9e-4 px in all. The angle is cross / dot:
# the 52 terms of cross move by at most sum (|u| + |v|) x 2 x 9e-4 (the sum is
# 360), dot is at least 0.75 x sum (u^2 + v^2) = 0.75 x 1704 for the depth
# changes drawn here.
ATOL_PX = 9e-4
ATOL_ANGLE = 360 * 2 * 9e-4 / (0.75 * 1704)


@pytest.mark.parametrize("cap,n_img", [(1, 1), (5, 3), (333, 2), (4096, 3)])
def test_lanes_equal_threads(cap, n_img):
    lim = 96 * torch.cuda.get_device_properties(0).multi_processor_count
    assert cap * n_img <= lim
    rng = np.random.default_rng(cap)
    big = lim // n_img + 4096               # a thread each
    pts = np.stack([rng.uniform(0, 1920, (n_img, big)), rng.uniform(0, 1080, (n_img, big))], 2)
    rho = rng.uniform(-0.05, 0.5, (n_img, big))
    kk = (900.0, 910.0, 955.0, 538.0)
    ang = 0.01 * rng.normal(size=(n_img, 3))
    poses = np.zeros((n_img, 12), np.float32)
    for i in range(n_img):
        wx, wy, wz = ang[i]
        poses[i, :9] = [1, -wz, wy, wz, 1, -wx, -wy, wx, 1]
        poses[i, 9:] = rng.uniform(-0.2, 0.2, 3)
    poses = torch.from_numpy(poses).cuda()
    pts = torch.from_numpy(pts.astype(np.float32)).cuda()
    rho = torch.from_numpy(rho.astype(np.float32)).cuda()

    def run(n, count):
        init = torch.full((n_img, n, 3), -1.0, device="cuda")
        valid = torch.full((n_img, n), 7, dtype=torch.uint8, device="cuda")
        vio.predict_warp(kk, kk, poses, pts[:, :n].contiguous(), rho[:, :n].contiguous(), count, n,
                         n_img, init, valid)
        torch.cuda.synchronize()
        return init, valid
    count = torch.full((n_img,), max(cap - 2, 1), dtype=torch.int32, device="cuda")
    live = int(count[0])
    a, va = run(cap, count)
    b, vb = run(big, None)
    assert torch.equal(va[:, :live], vb[:, :live]) and int(va[:, live:].sum()) == 0
    assert bool((a[:, live:] == -1).all())   # slots beyond the count are left
    d = (a[:, :live] - b[:, :live]).abs()
    assert float(d[..., :2].max()) <= ATOL_PX and float(d[..., 2].max()) <= ATOL_ANGLE
