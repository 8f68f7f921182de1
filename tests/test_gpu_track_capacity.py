"""Steps of a batch whose lists have far more room than tracks, and of the same
batch with little, bit for bit (the first run a warp per keypoint, however much
room there is)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")
from test_gpu_front_split import _frames  # noqa: E402


@pytest.mark.parametrize("ns,cell", [(1, 32), (7, 16)])   # below and above the groups' limit
def test_capacity_does_not_change_the_lists(ns, cell):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)
    w, h = 640, 480
    p = vio.default_params(n_levels=4, cell_w=cell, cell_h=cell)
    cells = (w // cell) * (h // cell)
    frames = [_frames(w, h, 3, 70 + s) for s in range(ns)]
    lists = []
    for cap in (2 * cells, 9000):
        b = vio.Batch([(p, w, h, ns, cap)])
        for t in range(3):
            for s in range(ns):
                b.next_frame(0, s).copy_(frames[s][t])
            b.step()
        torch.cuda.synchronize()
        lists.append([b.stream_lists(0, s) for s in range(ns)])
    for (xa, ia), (xb, ib) in zip(*lists):
        for c in range(2):
            assert len(ia[c]) > 0 and np.array_equal(ia[c], ib[c])
            assert np.array_equal(xa[c], xb[c])
