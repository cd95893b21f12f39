"""bench.py's issue-rate peak: from the clock sampled during the kernel's own timing,
and none without a sample."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_issue_rate_needs_a_sample():
    import bench
    assert bench.issue_rate(None, 152) is None
    assert bench.issue_rate({"sm_mhz": None}, 152) is None
    assert bench.issue_rate({"sm_mhz": 1500.0}, 152) == pytest.approx(4 * 152 * 1.5)


def test_no_clock_is_assumed():
    src = open(os.path.join(ROOT, "bench.py")).read()
    assert not re.search(r'sm_mhz.*or\s+\d', src)
    # the FP64 peak is that of the FP64 region
    assert "issue_rate(clk_step.summary()" in src


def test_regions_keep_their_own_samples():
    import bench
    a, b = bench.Clocks(0), bench.Clocks(0)
    line = "0, {}, 2070, 500.0, 0x0, Not Active, Not Active, Not Active, Not Active\n"
    for c, mhz in ((a, 1500), (b, 2070)):
        c.proc = True  # sampled
        with open(c.path, "w") as f:
            f.write(line.format(mhz) * 3)
    try:
        assert a.summary()["sm_mhz"] == 1500.0 and b.summary()["sm_mhz"] == 2070.0
    finally:
        os.remove(a.path)
        if os.path.exists(b.path):
            os.remove(b.path)
