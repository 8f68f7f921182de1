"""The grouped tracker's device code (track_group.cuh) run on the host under
AddressSanitizer, against the per-warp tracker bit for bit: both group sizes,
levels with word-aligned and unaligned rows, images small enough that most
windows touch an edge."""
import os
import shutil

import pytest

from test_emulated_kernels import CSRC, _build, _run


@pytest.mark.parametrize("lanes,w,h,levels,pitch,seed", [
    (4, 160, 120, 3, 160, 1),     # rows on 16-byte boundaries
    (4, 97, 75, 2, 97, 2),        # rows at any byte
    (16, 133, 90, 3, 136, 3),     # padded rows
    (16, 41, 33, 1, 41, 4),       # barely larger than a window
])
def test_groups_equal_the_warp_form(tmp_path, lanes, w, h, levels, pitch, seed):
    shutil.copy(os.path.join(CSRC, "track_group.cuh"), str(tmp_path / "track_group.cuh"))
    out = _run(_build(tmp_path, "trkg_check"), lanes, w, h, levels, pitch, seed)
    assert " ok 0 " not in out, out
