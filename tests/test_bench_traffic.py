"""The DRAM traffic that the bench line reports is the committed capture's (no GPU)."""
import os
import re

import pytest

import bench

CAPTURE = os.path.join(bench.ROOT, "profiles", "k_icp_sched_k_frontend_current.md")


@pytest.mark.parametrize("column, precision", enumerate(["fp32", "fp16"]))
def test_traffic_is_the_capture_s(column, precision):
    with open(CAPTURE) as f:
        text = f.read()

    def row(name):
        return int(re.search(rf"^\| {name}[^|]*\| (\d+) \| (\d+) \|$", text, re.M).group(column + 1))

    want = (row("bytes read") + row("bytes written")) / row("pixel-iterations of the launch")
    assert bench.NCU_DRAM_PER_PX_ITER[precision] == pytest.approx(want, rel=1e-12)
