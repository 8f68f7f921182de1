"""The grouped tracker's device code on the host (AddressSanitizer, against the
per-warp tracker bit for bit, as test_track_group_host.py) with starts of a
finite position and a non-finite angle at keypoints inside the image, with and
without steps to take."""
import os
import shutil

import pytest

from test_emulated_kernels import CSRC, EMU, _build, _run

LAST = "if (i == 15) { K.has_init = true; K.ith = 2.9f; }"
MORE = """
    if (i >= 16 && i < 28) {
      const float bad[3] = {nan, INFINITY, -INFINITY};
      K.px = 0.5f * (float)w + (float)(i % 4);
      K.py = 0.5f * (float)h - (float)(i % 3);
      K.has_init = true;
      K.ix = K.px + 0.5f;
      K.iy = K.py;
      K.ith = bad[i % 3];
      I.retry = i % 6 == 5;
    }"""


# four lanes per keypoint: the form that is launched
@pytest.mark.parametrize("w,h,levels,pitch,seed", [
    (160, 120, 3, 160, 5),
    (97, 75, 1, 97, 6),
])
def test_non_finite_start_angles(tmp_path, w, h, levels, pitch, seed):
    shutil.copy(os.path.join(CSRC, "track_group.cuh"), str(tmp_path / "track_group.cuh"))
    text = open(os.path.join(EMU, "trkg_check.cpp")).read()
    assert text.count(LAST) == 1
    (tmp_path / "trkg_angles.cpp").write_text(text.replace(LAST, LAST + MORE))
    out = _run(_build(tmp_path, str(tmp_path / "trkg_angles")), 4, w, h, levels, pitch, seed)
    assert " ok 0 " not in out, out
