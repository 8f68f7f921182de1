"""The half-row loads of the network input extraction (initnet_dev.cuh) run on
the host under AddressSanitizer, against plain byte reads: rows at every word
remainder, halves over and far beyond every edge."""
from test_emulated_kernels import _build, _run


def test_half_rows_on_host(tmp_path):
    _run(_build(tmp_path, "halfrow_check", ["-fwrapv"]))
