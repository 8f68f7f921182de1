"""The front of a large step as separate launches (a pyramid level each, then
the detection) against the fused launch, bit for bit: streams of odd sizes and
different level counts, one of them skipped in a step, plain and replayed
from a graph."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")

GROUPS = [  # w, h, n_streams, cell, levels
    (1281, 723, 2, 48, 5),
    (1000, 701, 1, 37, 3),
    (97, 65, 1, 20, 2),
]


def _frames(w, h, n, seed):
    g = torch.Generator().manual_seed(seed)
    t = torch.nn.functional.avg_pool2d(torch.rand((1, 1, h + 40, w + 60), generator=g), 5, 1, 2)
    t = ((t - 0.5) * 900 + 128).clamp(0, 255)[0, 0]
    out = torch.stack([torch.stack([t[i: i + h, 2 * i: 2 * i + w],
                                    t[i: i + h, 2 * i + 7: 2 * i + 7 + w]]) for i in range(n)])
    return out.to(torch.uint8).cuda()


@pytest.mark.parametrize("graph", [False, True])
def test_split_front_equals_fused(graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)
    groups, frames = [], []
    for gi, (w, h, ns, cell, L) in enumerate(GROUPS):
        p = vio.default_params(n_levels=L, cell_w=cell, cell_h=cell, round_mode=gi % 2)
        groups.append((p, w, h, ns, 2 * (w // cell) * (h // cell)))
        frames.append([_frames(w, h, 4, 10 * gi + s) for s in range(ns)])
    a, b = vio.Batch(groups), vio.Batch(groups)
    b.set_tune(128, 0, 0, 4, 256, 0)
    assert a.launches_per_step() == 3 + 4 and b.launches_per_step() == 3
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for batch in (a, b):
            batch.set_graph(graph)
            for t in range(4):
                act = [1, int(t != 2), 1, 1]
                k = 0
                for gi, g in enumerate(frames):
                    for s, f in enumerate(g):
                        if act[k]:
                            batch.next_frame(gi, s).copy_(f[t])
                        k += 1
                batch.step(act, stream=stream)
    stream.synchronize()
    for gi, (w, h, ns, cell, L) in enumerate(GROUPS):
        for s in range(ns):
            xa, ia = a.stream_lists(gi, s)
            xb, ib = b.stream_lists(gi, s)
            for c in range(2):
                assert len(ia[c]) > 0 and np.array_equal(ia[c], ib[c])
                assert np.array_equal(xa[c], xb[c])
