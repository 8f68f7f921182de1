"""The model-based start of a keypoint does not depend on the size of its launch:
eight lanes per keypoint against one thread per keypoint, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")


@pytest.mark.parametrize("cap,n_img", [(1, 1), (131, 3), (4096, 3)])
def test_lanes_equal_threads_bit_for_bit(cap, n_img):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)
    lim = 96 * torch.cuda.get_device_properties(0).multi_processor_count
    assert cap * n_img <= lim
    big = lim // n_img + 64                 # a thread each
    rng = np.random.default_rng(100 + cap)
    pts = rng.uniform(0, [1920, 1080], (n_img, big, 2)).astype(np.float32)
    rho = rng.uniform(-0.02, 0.5, (n_img, big)).astype(np.float32)
    poses = np.zeros((n_img, 12), np.float32)
    poses[:, :9] = np.eye(3).reshape(-1) + 0.05 * rng.normal(size=(n_img, 9))
    poses[:, 9:] = rng.normal(0, 0.3, (n_img, 3))
    pts, rho, poses = (torch.from_numpy(v).cuda() for v in (pts, rho, poses))

    def run(n):
        init = torch.zeros((n_img, n, 3), device="cuda")
        valid = torch.zeros((n_img, n), dtype=torch.uint8, device="cuda")
        vio.predict_warp((900.0, 910.0, 955.0, 538.0), (880.0, 905.0, 950.0, 541.0), poses,
                         pts[:, :n].contiguous(), rho[:, :n].contiguous(), None, n, n_img, init,
                         valid)
        return init.view(torch.int32), valid
    (a, va), (b, vb) = run(cap), run(big)
    assert torch.equal(va, vb[:, :cap])
    assert torch.equal(a, b[:, :cap])
