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
