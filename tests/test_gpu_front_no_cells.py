"""Streams whose image is smaller than one detection cell: their steps are
counted (the statistics are addressed by that count) whether the front of a step
is one launch or several, and with a single pyramid level."""
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


@pytest.mark.parametrize("groups", [
    [(1281, 723, 3, 48, 5), (97, 65, 2, 100, 2)],    # launches per level
    [(200, 151, 1, 32, 3), (97, 65, 1, 100, 1)],     # one launch, no pyramid tiles
    [(97, 65, 2, 100, 1)],                           # nothing else in the launch
])
def test_batch_steps_are_counted(groups):
    b = vio.Batch([(vio.default_params(n_levels=L, cell_w=c, cell_h=c), w, h, ns,
                    max(8, 2 * (w // c) * (h // c))) for w, h, ns, c, L in groups])
    frames = [[_frames(w, h, 3, 10 * gi + s) for s in range(ns)]
              for gi, (w, h, ns, c, L) in enumerate(groups)]
    for t in range(3):
        for gi, g in enumerate(frames):
            for s, f in enumerate(g):
                b.next_frame(gi, s).copy_(f[t])
        b.step()
    torch.cuda.synchronize()
    for gi, (w, h, ns, c, L) in enumerate(groups):
        ring, steps = b.read_stats(gi)
        assert steps == 3
        assert (ring[3:] == 0).all()
        for s in range(ns):
            xy, ids = b.stream_lists(gi, s)
            assert (len(ids[0]) > 0) == (c < w)


def test_frontend_steps_are_counted():
    fe = vio.Frontend(vio.default_params(n_levels=1, cell_w=100, cell_h=100), 97, 65, 1, 8)
    fe.run(_frames(97, 65, 3, 1)[:, None].contiguous())
    torch.cuda.synchronize()
    ring, steps = fe.read_stats()
    assert steps == 3 and (ring == 0).all()
