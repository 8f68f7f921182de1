"""A call whose launches the runtime refuses (its stream's capture was
invalidated) reports the error; the next call does not report it again."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

vio = pytest.importorskip("paper_2609_30459_gb300.vio")


@pytest.mark.parametrize("call", ["build", "detect"])
def test_error_is_reported_once(call):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    vio.load(build=True)
    w, h, L = 200, 150, 3
    frames = torch.randint(0, 256, (2, h, w), dtype=torch.uint8, device="cuda")
    ctx = vio.Context(vio.default_params(n_levels=L, cell_w=32, cell_h=32), w, h, 2)
    pyr = vio.Pyramids(frames, L)
    cap = (w // 32) * (h // 32)
    out = (torch.zeros((2, cap, 2), device="cuda"),
           torch.zeros((2, cap), dtype=torch.int16, device="cuda"),
           torch.zeros(2, dtype=torch.int32, device="cuda"))

    def run(stream=None):
        if call == "build":
            ctx.pyramid_build(pyr, stream=stream)
        else:
            ctx.detect_grid(pyr, pyr.batch(), *out, cap, stream=stream)
    run()
    torch.cuda.synchronize()
    # the runtime's own capture calls: a failed torch.cuda.graph would leave its
    # random generators in the capture
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    s, graph = torch.cuda.Stream(), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(ctypes.c_void_p(s.cuda_stream), 0) == 0
    assert rt.cudaDeviceSynchronize() != 0     # not allowed here: invalidates the capture
    with pytest.raises(vio.VioError):
        run(s)
    assert rt.cudaStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) != 0
    rt.cudaGetLastError()
    run()
    torch.cuda.synchronize()
    assert int(out[2].sum()) > 0 or call == "build"
